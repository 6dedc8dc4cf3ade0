// fp32-accumulate CUDA-core GEMMs.  They serve the fp32 workloads (whose 1e-4 tolerance a
// single-pass reduced-precision tensor-core product cannot meet; those shapes are tiny) and
// any shape the tensor-core path does not take.
#include <algorithm>

#include "kernels.h"

namespace ssm {

constexpr int TM = 64, TN = 64, TK = 16;
constexpr int kGemmThreads = 256;
constexpr long long kMaxGridZ = 65535;

template <typename T>
__device__ __forceinline__ void load4(const T* p, float (&v)[4]);
template <>
__device__ __forceinline__ void load4<float>(const float* p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <>
__device__ __forceinline__ void load4<__nv_bfloat16>(const __nv_bfloat16* p, float (&v)[4]) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
    const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
    v[0] = __low2float(lo); v[1] = __high2float(lo); v[2] = __low2float(hi); v[3] = __high2float(hi);
}

template <typename T>
__device__ __forceinline__ void store4(T* p, const float (&v)[4]);
template <>
__device__ __forceinline__ void store4<float>(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, const float (&v)[4]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

struct EpiArgs {
    void* out;
    const float* diag;
    const void* skip;
    const void* add;
    int ldo;
};

// out[m,n] = sum_k A[m,k] Bm[n,k]; both operands K-contiguous.  K % 4 == 0.
// TO: type of out; TS: type of the skip operand; the addend, where there is one, is fp32.
template <typename TA, typename TB, typename TO, typename TS, bool kAddDiag>
__global__ void __launch_bounds__(kGemmThreads)
gemm_tn_kernel(const TA* A, int lda, const TB* Bm, int ldb, int M, int N, int K,
               EpiArgs e) {
    grid_dep_wait();
    __shared__ __align__(16) float As[TK][TM + 4];
    __shared__ __align__(16) float Bs[TK][TN + 4];
    const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;   // rows along x: grid.y is limited to 65535
    const int tid = threadIdx.x;
    const int lr = tid >> 2;         // 0..63: row of the tile this thread loads
    const int lk = (tid & 3) * 4;    // 0,4,8,12: k offset
    const int tx = tid & 15, ty = tid >> 4;  // 16 x 16 threads, 4 x 4 outputs each
    float acc[4][4] = {};
    float va[4], vb[4];
    auto fetch = [&](int k0) {   // the next block's operands, on their way while this one is multiplied
#pragma unroll
        for (int i = 0; i < 4; ++i) va[i] = vb[i] = 0.f;
        if (m0 + lr < M && k0 + lk < K) load4<TA>(A + (size_t)(m0 + lr) * lda + k0 + lk, va);
        if (n0 + lr < N && k0 + lk < K) load4<TB>(Bm + (size_t)(n0 + lr) * ldb + k0 + lk, vb);
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            As[lk + i][lr] = va[i];
            Bs[lk + i][lr] = vb[i];
        }
        __syncthreads();
        if (k0 + TK < K) fetch(k0 + TK);
#pragma unroll
        for (int k = 0; k < TK; ++k) {
            const float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
            const float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    // Not earlier: the next kernel's blocks would be placed while this one's fill the SMs unevenly, and with several blocks
    // per SM that imbalance lasted (6272 x 176 x 168: 17 -> 28 us).
    grid_dep_launch();
    // 4 neighbouring columns at a time (N is a multiple of 8); everything is read before anything is written
    const int n = n0 + tx * 4;
    if (n >= N) return;
    if (kAddDiag) {
        const float4 dg = *reinterpret_cast<const float4*>(e.diag + n);
        float sk[4][4], ad[4][4] = {};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = m0 + ty * 4 + i;
            if (m >= M) continue;
            load4<TS>(reinterpret_cast<const TS*>(e.skip) + (size_t)m * e.ldo + n, sk[i]);
            if (e.add) load4<float>(reinterpret_cast<const float*>(e.add) + (size_t)m * e.ldo + n, ad[i]);
        }
        const float dd[4] = {dg.x, dg.y, dg.z, dg.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(dd[j], sk[i][j], acc[i][j]) + ad[i][j];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m < M) store4<TO>(reinterpret_cast<TO*>(e.out) + (size_t)m * e.ldo + n, acc[i]);
    }
}

template <typename TA, typename TB>
static void dispatch_tn(const GemmTN& g, cudaStream_t st) {
    dim3 grid((g.M + TM - 1) / TM, (g.N + TN - 1) / TN);
    count_launch();
    EpiArgs e{g.out, g.diag, g.skip, g.add, g.N};
    const TA* A = (const TA*)g.A;
    const TB* Bm = (const TB*)g.Bm;
    using bf = __nv_bfloat16;
    if (g.epi == Epi::StoreF32)
        launch_dep(gemm_tn_kernel<TA, TB, float, float, false>, grid, kGemmThreads, 0, st, A, g.lda, Bm, g.ldb, g.M, g.N, g.K, e);
    else if (g.out_bf16 && g.skip_bf16)
        launch_dep(gemm_tn_kernel<TA, TB, bf, bf, true>, grid, kGemmThreads, 0, st, A, g.lda, Bm, g.ldb, g.M, g.N, g.K, e);
    else if (g.out_bf16)
        launch_dep(gemm_tn_kernel<TA, TB, bf, float, true>, grid, kGemmThreads, 0, st, A, g.lda, Bm, g.ldb, g.M, g.N, g.K, e);
    else if (g.skip_bf16)
        launch_dep(gemm_tn_kernel<TA, TB, float, bf, true>, grid, kGemmThreads, 0, st, A, g.lda, Bm, g.ldb, g.M, g.N, g.K, e);
    else
        launch_dep(gemm_tn_kernel<TA, TB, float, float, true>, grid, kGemmThreads, 0, st, A, g.lda, Bm, g.ldb, g.M, g.N, g.K, e);
}

void launch_gemm_tn(const GemmTN& g, cudaStream_t st) {
    if (g.a_bf16 && g.b_bf16) dispatch_tn<__nv_bfloat16, __nv_bfloat16>(g, st);
    else if (g.a_bf16) dispatch_tn<__nv_bfloat16, float>(g, st);
    else if (g.b_bf16) dispatch_tn<float, __nv_bfloat16>(g, st);
    else dispatch_tn<float, float>(g, st);
}

// part[s,i,j] = sum_{k in slice s} A[k,i] Bm[k,j]; both operands contiguous in i / j, Bm fp32.  Up to two products of one
// shape (blockIdx.z = product * splits + slice) and, behind them, the column dot products of a and b: a layer's weight
// gradients and dD in one launch, which at the sizes this path is for are a few microseconds each.
struct NtSimtArgs {
    GemmNT g[2];
    int n, k_per_split;
    const void *dot_a, *dot_b;
    bool dot_a_bf16, dot_b_bf16;
    float* dot_part;
    int dot_groups;               // row groups
    long long dot_blocks;         // row groups x 128-column blocks: the blocks behind the products take them in turn
};

__device__ __forceinline__ void load4_any(const void* p, bool bf16, size_t i, float (&v)[4]) {
    if (bf16) load4<__nv_bfloat16>(reinterpret_cast<const __nv_bfloat16*>(p) + i, v);
    else load4<float>(reinterpret_cast<const float*>(p) + i, v);
}

// kChains: rows are summed in chains of 8 before they are added to the rest, as the one-kernel passes of small layers do.
template <bool kChains>
__global__ void __launch_bounds__(kGemmThreads)
gemm_nt_kernel(const __grid_constant__ NtSimtArgs q) {
    grid_dep_wait();
    __shared__ __align__(16) float As[TK][TM + 4];
    __shared__ __align__(16) float Bs[TK][TN + 4];
    const int z = (int)blockIdx.z / q.g[0].splits;
    if (z >= q.n) {   // dot products: block = 32 column quads x 8 row lanes, kDotRows rows at a time
        const int per_z = (int)(gridDim.x * gridDim.y), first_z = q.n * q.g[0].splits;
        const int C = q.g[0].I, M = q.g[0].K, rl = threadIdx.x >> 5;
        float4(*sm)[32] = reinterpret_cast<float4(*)[32]>(&As[0][0]);   // 8 x 32 float4 = 4 KB
        static_assert(sizeof(As) >= 8 * 32 * sizeof(float4), "the dot products' sums fit the operand tile");
        grid_dep_launch();
        for (long long blk = (long long)((int)blockIdx.z - first_z) * per_z + (int)(blockIdx.y * gridDim.x + blockIdx.x); blk < q.dot_blocks;
             blk += (long long)((int)gridDim.z - first_z) * per_z) {
            const int grp = (int)(blk % q.dot_groups), c = (int)(blk / q.dot_groups * 32 + (threadIdx.x & 31)) * 4;
            const int r0 = grp * kDotRows, r1 = min(M, r0 + kDotRows);
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            if (c < C) {
#pragma unroll 4
                for (int r = r0 + rl; r < r1; r += 8) {
                    float va[4], vb[4];
                    load4_any(q.dot_a, q.dot_a_bf16, (size_t)r * C + c, va);
                    load4_any(q.dot_b, q.dot_b_bf16, (size_t)r * C + c, vb);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i] = fmaf(va[i], vb[i], acc[i]);
                }
            }
            __syncthreads();   // the sums of the group before have been read
            sm[rl][threadIdx.x & 31] = make_float4(acc[0], acc[1], acc[2], acc[3]);
            __syncthreads();
            if (rl == 0 && c < C) {
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = sm[i][threadIdx.x];
                    t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
                }
                *reinterpret_cast<float4*>(q.dot_part + (size_t)grp * C + c) = t;
            }
        }
        return;
    }
    const GemmNT& g = q.g[z];
    const int slice = (int)blockIdx.z - z * g.splits, I = g.I, J = g.J;
    const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const int kb = slice * q.k_per_split, ke = min(g.K, kb + q.k_per_split);
    const int tid = threadIdx.x;
    const int lk = tid >> 4;          // 0..15
    const int lc = (tid & 15) * 4;    // 0..60
    const int tx = tid & 15, ty = tid >> 4;
    float acc[4][4] = {};
    float va[4], vb[4];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) va[i] = vb[i] = 0.f;
        if (k0 + lk < ke) {
            if (i0 + lc < I) load4_any(g.A, g.a_bf16, (size_t)(k0 + lk) * I + i0 + lc, va);
            if (j0 + lc < J) load4<float>(g.Bm + (size_t)(k0 + lk) * J + j0 + lc, vb);
        }
    };
    fetch(kb);
    for (int k0 = kb; k0 < ke; k0 += TK) {
        *reinterpret_cast<float4*>(&As[lk][lc]) = make_float4(va[0], va[1], va[2], va[3]);
        *reinterpret_cast<float4*>(&Bs[lk][lc]) = make_float4(vb[0], vb[1], vb[2], vb[3]);
        __syncthreads();
        if (k0 + TK < ke) fetch(k0 + TK);
        constexpr int kChain = kChains ? 8 : TK;
#pragma unroll
        for (int k1 = 0; k1 < TK; k1 += kChain) {
            float part[4][4] = {};
            float(&to)[4][4] = kChains ? part : acc;
#pragma unroll
            for (int k = k1; k < k1 + kChain; ++k) {
                const float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
                const float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
                const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) to[i][j] = fmaf(av[i], bv[j], to[i][j]);
            }
            if (kChains)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] += part[i][j];
        }
        __syncthreads();
    }
    grid_dep_launch();
    float* out = g.part + (size_t)slice * I * J;
    const int jj = j0 + tx * 4;
    if (jj >= J) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int ii = i0 + ty * 4 + i;
        if (ii < I) store4<float>(out + (size_t)ii * J + jj, acc[i]);
    }
}

// Slices of the rows: about three blocks per SM for a pair of products, at least 64 rows each (6272 rows, 168 x 176
// outputs: one launch of 468 blocks 38 us, two of 117 59 us), and at most 512 rows as long as there are 64 slices or
// fewer: a slice is one chain of fp32 additions, and one of L rows is off by about sqrt(L / 6) 2^-24 of its sum.  A gate
// of 12800 x 1024 as one chain per output 2543 us with dW 2.0e-6 off (elements to 1.1e-4), in 25 slices 2396 us and
// 4.4e-7 (2.9e-5); a layer of 32000 rows at 520, 264 with bf16 I/O 4012 / 3506 us, dB 2.3e-6 / 6.2e-7.
int gemm_nt_splits(int K, int I, int J) {
    const int tiles = ((J + TN - 1) / TN) * ((I + TM - 1) / TM);
    const int want = 3 * device_sm_count() / (2 * tiles), most = (K + 63) / 64, least = (K + 511) / 512;
    return std::max(1, std::min(std::max(std::min(want, most), least), 64));
}

void launch_gemm_nt(const GemmNT* g, int n, const SimtDot* dot, cudaStream_t st, bool short_chains) {
    NtSimtArgs q{};
    for (int i = 0; i < n; ++i) q.g[i] = g[i];
    q.n = n;
    const int kps = (g->K + g->splits - 1) / g->splits;
    q.k_per_split = (kps + TK - 1) / TK * TK;
    dim3 grid((g->J + TN - 1) / TN, (g->I + TM - 1) / TM, n * g->splits);
    if (dot) {
        q.dot_a = dot->a, q.dot_b = dot->b, q.dot_a_bf16 = dot->a_bf16, q.dot_b_bf16 = dot->b_bf16, q.dot_part = dot->part;
        q.dot_groups = dot_groups(g->K);
        q.dot_blocks = (long long)q.dot_groups * ((g->I + 127) / 128);
        // (a grid has at most 65535 blocks along z: from 8.4 million rows of one output tile on a block takes several groups)
        const long long per_z = (long long)grid.x * grid.y;
        grid.z += (unsigned)std::min<long long>((q.dot_blocks + per_z - 1) / per_z, kMaxGridZ - grid.z);
    }
    count_launch();
    launch_dep(short_chains ? gemm_nt_kernel<true> : gemm_nt_kernel<false>, grid, kGemmThreads, 0, st, q);
}

}  // namespace ssm
