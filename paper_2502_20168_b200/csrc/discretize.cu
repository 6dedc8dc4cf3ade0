// Zero-order-hold discretisation of the diagonal SSM (Sec. III-B, Eq. 3) and its adjoint,
// plus the packing of the discretised parameters into real GEMM operands.
#include <algorithm>

#include "kernels.h"
#include "zoh.cuh"

namespace ssm {

// One block per state p: Abar[p], Bbar[p, :] = gamma_p * B[p, :].
__global__ void discretize_kernel(int H, const float2* Lambda, const float* Delta,
                                  const float2* Bc, float2* Abar, float2* Bbar) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float2 gamma_s;
    const int p = blockIdx.x;
    if (threadIdx.x == 0) {
        ZohTerms z = zoh_terms(Lambda[p], Delta[p]);
        Abar[p] = make_float2((float)z.ar, (float)z.ai);
        gamma_s = make_float2((float)z.gr, (float)z.gi);
    }
    __syncthreads();
    const float2 g = gamma_s;
    for (int h = threadIdx.x; h < H; h += blockDim.x) Bbar[(size_t)p * H + h] = cmul(g, Bc[(size_t)p * H + h]);
}

// ssm_discretize_bwd: one block per state p.
__global__ void discretize_bwd_kernel(int H, int P, const float2* Lambda, const float* Delta,
                                      const float2* Bc, const float2* gAbar,
                                      const float2* gBbar, float2* dLambda,
                                      float* dDelta, float2* dB) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float2 gamma_s;
    __shared__ float red[2][32];
    const int p = blockIdx.x;
    const float2 lam = Lambda[p];
    const float dt = Delta[p];
    ZohTerms z = {};
    if (threadIdx.x == 0) {
        z = zoh_terms(lam, dt);
        gamma_s = make_float2((float)z.gr, (float)z.gi);
    }
    __syncthreads();
    const float2 gc = cconj(gamma_s);
    float sr = 0.f, si = 0.f;  // g_gamma = sum_h conj(B) gBbar
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
        float2 gb = gBbar[(size_t)p * H + h];
        float2 b = Bc[(size_t)p * H + h];
        dB[(size_t)p * H + h] = cmul(gc, gb);
        float2 t = cmul(cconj(b), gb);
        sr += t.x;
        si += t.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = sr;
        red[1][threadIdx.x >> 5] = si;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ggr = 0.0, ggi = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            ggr += red[0][w];
            ggi += red[1][w];
        }
        zoh_adjoint(z, lam, dt, gAbar[p].x, gAbar[p].y, ggr, ggi, dLambda[p], dDelta[p]);
    }
}

// hi = bf16(w) and lo = bf16(w - hi) into row n of the hi block and of the lo block of a stacked operand of
// 2^stack_log2 rows per block.
__device__ __forceinline__ void store_split(__nv_bfloat16* W, int H, int n, int h, float w, int stack_log2) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(w);
    const __nv_bfloat16 lo = __float2bfloat16_rn(w - __bfloat162float(hi));
    const int stack = 1 << stack_log2;
    const size_t r = (size_t)(((n >> stack_log2) << (stack_log2 + 1)) + (n & (stack - 1)));
    W[r * H + h] = hi;
    W[(r + stack) * H + h] = lo;
}

// The three bf16 planes of v (hi + mid + lo = v), `plane_stride` elements apart.
__device__ __forceinline__ void store3(__nv_bfloat16* base, size_t plane_stride, float v) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    base[0] = hi;
    base[plane_stride] = mid;
    base[2 * plane_stride] = __float2bfloat16_rn(r1 - __bfloat162float(mid));
}
__device__ __forceinline__ void store3_pair(float a, float b, __nv_bfloat162& hi, __nv_bfloat162& mid, __nv_bfloat162& lo) {
    hi = __floats2bfloat162_rn(a, b);
    const float2 h = __bfloat1622float2(hi);
    const float a1 = a - h.x, b1 = b - h.y;
    mid = __floats2bfloat162_rn(a1, b1);
    const float2 m = __bfloat1622float2(mid);
    lo = __floats2bfloat162_rn(a1 - m.x, b1 - m.y);
}

// ---------------------------------------------------------------------------------------------
// Discretisation and the packed projection operands of a layer, one kernel
// ---------------------------------------------------------------------------------------------
// From Lambda, Delta, B, C: Abar (as an fp32 pair) and the operands of the four projections, which are Bbar and
// C once with the states along the rows (h contiguous: weights of Bu and g_x) and once with h along the rows
// (states contiguous: weights of du and y).  A block owns 32 states x 32 features: it reads its tile of B
// (rows of 32 h) and of C (rows of 32 states), turns both round in shared memory, so that every global access of
// a warp is a run of 64 to 256 contiguous bytes, and evaluates gamma of its 32 states in double precision, one
// per lane of a warp.  Blocks that own the same states repeat that evaluation (about 1.5 us, the length of the
// tile's own loads).  What bounds it is latency: H x P weights are 1 - 8 MB in and out.  H = 512, P = 256: bf16
// halves 7.6 -> 4.6 us, planes 20.7 -> 4.4 us against one block per state with strided 2-byte accesses.
// kMode:
//   kPackTc     bf16 operands.  In the two projections that feed the states a weight w is carried as
//               hi = bf16(w), lo = bf16(w - hi), so that the states see ~16 mantissa bits of the parameters:
//               logical row n of the [2P, H] operand goes to rows (n/S) 2S + n%S (hi) and S further (lo) of the
//               stacked [4P, H] matrix (o.WB, o.WC).  S = 128 and n = 2p + c, or, for the kernels that scan in
//               their epilogue (group = states per chain), S = 2 group and the rows of two neighbouring states
//               interleaved as (re, re, im, im).  o.Cp, o.Bq: [H, 2P] single bf16.
//   kPackPlanes three bf16 planes of every operand side by side along its contraction index:
//               WB[2p+c, a H + h], WC likewise ([2P, 3H]);  Cp[h, a 2P + 2p+c], Bq likewise ([H, 3 2P]).
//   kPackF32    fp32: WB[2p+c, h], WC[2p+c, h] ([2P, H]);  Cp[h, 2p+c], Bq[h, 2p+c] ([H, 2P]).
// with c = 0 / 1 for Re / Im of Bbar and Re / -Im of C.  `hdr` (may be NULL): its status word is cleared.
enum PackMode { kPackTc, kPackPlanes, kPackF32 };
// A launch does the layers of a stack together (blockIdx.z), up to kN = kLayerBatch of them; a single layer's launch
// carries the parameters of one (kN = 1).
template <int kN>
struct PackArgs {
    PackJob job[kN];
    WsHeader* hdr;
    int group_log2;   // 0: no groups
};

template <int kMode>
__device__ __forceinline__ void store_row_pair(void* W, int H, int P, int group_log2, int p, int h, float re, float im) {
    if (kMode == kPackF32) {
        float* w = reinterpret_cast<float*>(W) + (size_t)(2 * p) * H + h;
        w[0] = re;
        w[H] = im;
    } else if (kMode == kPackPlanes) {
        __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(W) + (size_t)(2 * p) * 3 * H + h;
        store3(w, H, re);
        store3(w + 3 * (size_t)H, H, im);
    } else {
        // (all block sizes are powers of two: shifts, the divisions were most of this kernel's instructions)
        const int sl = group_log2 ? group_log2 + 1 : 7, in_group = p & ((1 << group_log2) - 1);
        const int n = group_log2 ? ((p >> group_log2) << sl) + 4 * (in_group >> 1) + (p & 1) : 2 * p;
        store_split(reinterpret_cast<__nv_bfloat16*>(W), H, n, h, re, sl);
        store_split(reinterpret_cast<__nv_bfloat16*>(W), H, n + (group_log2 ? 2 : 1), h, im, sl);
    }
}
template <int kMode>
__device__ __forceinline__ void store_col_pair(void* W, int P, int p, int h, float re, float im) {
    if (kMode == kPackF32) {
        reinterpret_cast<float2*>(W)[(size_t)h * P + p] = make_float2(re, im);
    } else if (kMode == kPackTc) {
        reinterpret_cast<__nv_bfloat162*>(W)[(size_t)h * P + p] = __floats2bfloat162_rn(re, im);
    } else {
        __nv_bfloat162 hi, mid, lo;
        store3_pair(re, im, hi, mid, lo);
        __nv_bfloat162* w = reinterpret_cast<__nv_bfloat162*>(W) + (size_t)h * 3 * P + p;
        w[0] = hi;
        w[P] = mid;
        w[2 * (size_t)P] = lo;
    }
}

template <int kMode, int kN>
__global__ void __launch_bounds__(256)
pack_params_kernel(int H, int P, const __grid_constant__ PackArgs<kN> o) {
    grid_dep_wait();
    grid_dep_launch();
    const PackJob& q = o.job[blockIdx.z];
    const float2 *Bc = q.Bc, *Cc = q.Cc;
    __shared__ float2 gamma_s[32];
    __shared__ float2 tB[32][33], tC[32][33];   // tB[state][h], tC[h][state]
    const int p_blocks = (P + 31) / 32, h_tile = (int)blockIdx.x / p_blocks;
    const int p0 = ((int)blockIdx.x - h_tile * p_blocks) * 32, h0 = h_tile * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float2 zero = make_float2(0.f, 0.f);
    float2 b[4], c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = w + 8 * i;
        b[i] = (p0 + r < P && h0 + lane < H) ? Bc[(size_t)(p0 + r) * H + h0 + lane] : zero;
        c[i] = (p0 + lane < P && h0 + r < H) ? Cc[(size_t)(h0 + r) * P + p0 + lane] : zero;
    }
    if (w == 0 && p0 + lane < P) {
        const int p = p0 + lane;
        const ZohTerms z = zoh_terms(q.Lambda[p], q.Delta[p]);
        gamma_s[lane] = make_float2((float)z.gr, (float)z.gi);
        if (h_tile == 0) {
            const float2 ah = make_float2((float)z.ar, (float)z.ai);
            q.Abar[p] = ah;
            q.Alo[p] = make_float2((float)(z.ar - (double)ah.x), (float)(z.ai - (double)ah.y));
            if (kMode == kPackTc && o.group_log2) {
                double re = z.ar, im = z.ai;
#pragma unroll
                for (int n = 2; n <= 128; n *= 2) {
                    const double r2 = re * re - im * im;
                    im = 2.0 * re * im;
                    re = r2;
                    if (n == 16 || n == 128) {
                        float* to = q.Apow + (size_t)(n == 16 ? 0 : 2) * P + 4 * (p >> 1) + (p & 1);
                        to[0] = (float)re;
                        to[2] = (float)im;
                    }
                }
            }
        }
    }
    if (threadIdx.x == 32 && blockIdx.x == 0 && blockIdx.z == 0 && o.hdr) o.hdr->status = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = w + 8 * i;
        b[i] = cmul(gamma_s[r], b[i]);
        tB[r][lane] = b[i];
        tC[r][lane] = c[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = w + 8 * i;
        if (p0 + r < P && h0 + lane < H) {   // state p0 + r, feature h0 + lane
            const float2 cc = tC[lane][r];
            store_row_pair<kMode>(q.WB, H, P, o.group_log2, p0 + r, h0 + lane, b[i].x, b[i].y);
            store_row_pair<kMode>(q.WC, H, P, o.group_log2, p0 + r, h0 + lane, cc.x, -cc.y);
        }
        if (p0 + lane < P && h0 + r < H) {   // state p0 + lane, feature h0 + r
            const float2 bb = tB[lane][r];
            store_col_pair<kMode>(q.Bq, P, p0 + lane, h0 + r, bb.x, bb.y);
            store_col_pair<kMode>(q.Cp, P, p0 + lane, h0 + r, c[i].x, -c[i].y);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Last sums of a layer's backward pass (the layers of a stack together)
// ---------------------------------------------------------------------------------------------
template <int kN>
struct TailArgs {
    GradTail layer[kN];
};
// The split-K partials of the weight-gradient products, part_b[s, h, 2p+c] (gBbar) and part_c[s, h, 2p+c] (dC, its
// imaginary columns negated), are added in order of s.  gBbar itself is not stored: it leaves as
// dB = conj(gamma) gBbar and as the sums g_gamma = sum conj(B) gBbar over the block's 32 features
// (gg_part[h / 32, p]).  A block owns 32 features x 32 states of one of the two matrices (blockIdx.z); gBbar is
// turned round in shared memory for the state-major dB.  Bound by reading the partials (L2 for small problems); with
// the sum and the state-major store as separate strided kernels a step spent 7.7 - 20 us here, now 7 - 10 us.
// kReduceWarps warps share the block's rows (one more evaluates gamma): 16 where there are many partials to add per
// element, else 8 (1024 x 1024 with 2 partials: 8.2 against 10.5 us; 512 x 512 with 9: 7.2 with 16 against 8.5).
template <int kReduceWarps, int kN>
__global__ void __launch_bounds__(32 * kReduceWarps + 32)
reduce_weight_grads_kernel(int H, int P, int splits, const __grid_constant__ TailArgs<kN> args) {
    grid_dep_wait();
    grid_dep_launch();
    const GradTail& q = args.layer[blockIdx.z >> 1];
    __shared__ float2 gamma_s[32];
    __shared__ float2 t[32][33];   // [feature][state]
    constexpr int kRows = 32 / kReduceWarps;
    const int p_blocks = (P + 31) / 32, h_tile = (int)blockIdx.x / p_blocks;
    const int p0 = ((int)blockIdx.x - h_tile * p_blocks) * 32, h0 = h_tile * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool is_c = (blockIdx.z & 1) != 0, p_ok = p0 + lane < P;
    if (w == kReduceWarps) {
        if (!is_c && p_ok) {
            const ZohTerms z = zoh_terms(q.Lambda[p0 + lane], q.Delta[p0 + lane]);
            gamma_s[lane] = make_float2((float)z.gr, (float)z.gi);
        }
        __syncthreads();
        return;
    }
    const float2* part = reinterpret_cast<const float2*>(is_c ? q.part_c : q.part_b);
    const size_t n = (size_t)H * P;   // complex values per split
    float2 acc[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) acc[i] = make_float2(0.f, 0.f);
    if (p_ok) {
        const float2* src = part + (size_t)(h0 + w) * P + p0 + lane;
#pragma unroll 8
        for (int s = 0; s < splits; ++s, src += n) {
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (h0 + w + kReduceWarps * i < H) acc[i] = cadd(acc[i], ld_stream(src + (size_t)kReduceWarps * i * P));
        }
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        if (is_c && p_ok && h0 + w + kReduceWarps * i < H)
            q.dC[(size_t)(h0 + w + kReduceWarps * i) * P + p0 + lane] = cconj(acc[i]);
        t[w + kReduceWarps * i][lane] = acc[i];
    }
    __syncthreads();
    if (is_c) return;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        const int pl = w + kReduceWarps * i, p = p0 + pl, h = h0 + lane;
        if (p >= P) continue;   // (the same for the whole warp)
        const float2 gb = t[lane][pl];
        float2 gq = make_float2(0.f, 0.f);
        if (h < H) {
            q.dB[(size_t)p * H + h] = cmul(cconj(gamma_s[pl]), gb);
            gq = cmul(cconj(q.Bc[(size_t)p * H + h]), gb);
        }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            gq.x += __shfl_xor_sync(0xffffffffu, gq.x, m);
            gq.y += __shfl_xor_sync(0xffffffffu, gq.y, m);
        }
        if (lane == 0) q.gg[(size_t)h_tile * P + p] = gq;
    }
}

// Adjoint of the discretisation with the sums of gAbar (gA_rows rows of [P]), g_gamma (gg_rows rows of [P]) and dD
// (dD_rows rows of [H]) folded in, in a fixed order.  A block owns 32 columns, its 32 warps take the rows in turn
// (the rows of partial sums are up to 512, the columns a few hundred: latency is all there is), one warp evaluates
// the P-sized double-precision terms meanwhile.  H = 512, P = 256: 6.2 - 9.5 -> 3.0 - 6.3 us (4 - 512 rows) against one block per state.
template <int kN>
__global__ void __launch_bounds__(1024)
layer_finalize_kernel(int H, int P, int gA_rows, int gg_rows, const __grid_constant__ TailArgs<kN> args) {
    grid_dep_wait();
    grid_dep_launch();
    const GradTail& q = args.layer[blockIdx.z];
    const float2 *Lambda = q.Lambda, *gA_part = q.gA_part, *gg_part = q.gg;
    const float* Delta = q.Delta;
    __shared__ double sA[2][32][33], sG[2][32][33];
    __shared__ ZohTerms zs[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p_blocks = (P + 31) / 32;
    if ((int)blockIdx.x >= p_blocks) {   // 32 columns of one of the sums over row groups (dD, then a stack's dw, db)
        double(*sD)[33] = sA[0];
        const int h_blocks = (H + 31) / 32, blk = (int)blockIdx.x - p_blocks, which = blk / h_blocks;
        const int h = (blk - which * h_blocks) * 32 + lane;
        const float* part = q.sum_part[which];
        double acc = 0.0;
        if (h < H)
            for (int r = w; r < q.sum_rows[which]; r += 32) acc += (double)part[(size_t)r * H + h];
        sD[w][lane] = acc;
        __syncthreads();
        if (w == 0 && h < H) {
            double t = 0.0;
#pragma unroll
            for (int i = 0; i < 32; ++i) t += sD[i][lane];
            q.sum_out[which][h] = (float)t;
        }
        return;
    }
    const int p = (int)blockIdx.x * 32 + lane;
    double ar = 0.0, ai = 0.0, gr = 0.0, gi = 0.0;
    if (p < P) {
#pragma unroll 4
        for (int r = w; r < gA_rows; r += 32) {
            const float2 v = gA_part[(size_t)r * P + p];
            ar += (double)v.x;
            ai += (double)v.y;
        }
        for (int r = w; r < gg_rows; r += 32) {
            const float2 v = gg_part[(size_t)r * P + p];
            gr += (double)v.x;
            gi += (double)v.y;
        }
        if (w == 31) zs[lane] = zoh_terms(Lambda[p], Delta[p]);
    }
    sA[0][w][lane] = ar;
    sA[1][w][lane] = ai;
    sG[0][w][lane] = gr;
    sG[1][w][lane] = gi;
    __syncthreads();
    // warps 0 .. 3 add one of the four sums each
    if (w < 4) {
        double(*src)[33] = w < 2 ? sA[w] : sG[w - 2];
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < 32; ++i) t += src[i][lane];
        src[0][lane] = t;
    }
    __syncthreads();
    if (w == 0 && p < P)
        zoh_adjoint(zs[lane], Lambda[p], Delta[p], sA[0][0][lane], sA[1][0][lane], sG[0][0][lane], sG[1][0][lane],
                    q.dLambda[p], q.dDelta[p]);
}

// One block per 32 x 32 tile, the tiles of 32 features after one another along x (y is limited to 65535 blocks).
static dim3 weight_tiles(int H, int P, int z) { return dim3((unsigned)((P + 31) / 32) * (unsigned)((H + 31) / 32), 1, z); }

template <int kMode, int kN>
static void launch_pack_n(int H, int P, int n, const PackJob* jobs, int group, WsHeader* hdr, cudaStream_t st) {
    PackArgs<kN> o{};
    std::copy(jobs, jobs + n, o.job);
    o.hdr = hdr;
    o.group_log2 = group == 64 ? 6 : (group == 32 ? 5 : 0);
    count_launch();
    launch_dep(pack_params_kernel<kMode, kN>, weight_tiles(H, P, n), 256, 0, st, H, P, o);
}
template <int kMode>
static void launch_pack(int H, int P, int n, const PackJob* jobs, int group, WsHeader* hdr, cudaStream_t st) {
    if (n == 1) return launch_pack_n<kMode, 1>(H, P, 1, jobs, group, hdr, st);
    for (int l = 0; l < n; l += kLayerBatch)
        launch_pack_n<kMode, kLayerBatch>(H, P, std::min(kLayerBatch, n - l), jobs + l, group, l == 0 ? hdr : nullptr, st);
}

void launch_discretize_pack_tc(int H, int P, int group, const PackJob& job, WsHeader* hdr, cudaStream_t st) {
    launch_pack<kPackTc>(H, P, 1, &job, group, hdr, st);
}
void launch_discretize_pack_planes(int H, int P, int n, const PackJob* jobs, WsHeader* hdr, cudaStream_t st) {
    launch_pack<kPackPlanes>(H, P, n, jobs, 0, hdr, st);
}
void launch_discretize_pack_f32(int H, int P, int n, const PackJob* jobs, WsHeader* hdr, cudaStream_t st) {
    launch_pack<kPackF32>(H, P, n, jobs, 0, hdr, st);
}

void launch_discretize(int H, int P, const float2* Lambda, const float* Delta, const float2* Bc, float2* Abar,
                       float2* Bbar, cudaStream_t st) {
    count_launch();
    launch_dep(discretize_kernel, P, 128, 0, st, H, Lambda, Delta, Bc, Abar, Bbar);
}

void launch_discretize_bwd(int H, int P, const float2* Lambda, const float* Delta, const float2* Bc,
                           const float2* gAbar, const float2* gBbar, float2* dLambda, float* dDelta, float2* dB,
                           cudaStream_t st) {
    count_launch();
    launch_dep(discretize_bwd_kernel, P, 128, 0, st, H, P, Lambda, Delta, Bc, gAbar, gBbar, dLambda, dDelta, dB);
}

int gamma_part_rows(int H) { return (H + 31) / 32; }

template <int kN>
static void launch_tail_n(int H, int P, int splits, int n, const GradTail* tails, int gA_rows, cudaStream_t st) {
    TailArgs<kN> args{};
    std::copy(tails, tails + n, args.layer);
    const int n_sums = tails[0].sum_out[2] ? 3 : 1;
    const dim3 grid = weight_tiles(H, P, 2 * n);
    count_launch(2);
    if (splits > 4) launch_dep(reduce_weight_grads_kernel<16, kN>, grid, 32 * 17, 0, st, H, P, splits, args);
    else launch_dep(reduce_weight_grads_kernel<8, kN>, grid, 32 * 9, 0, st, H, P, splits, args);
    launch_dep(layer_finalize_kernel<kN>, dim3((P + 31) / 32 + n_sums * ((H + 31) / 32), 1, n), 1024, 0, st, H, P, gA_rows,
               gamma_part_rows(H), args);
}

void launch_layer_tail(int H, int P, int splits, int n, const GradTail* tails, int gA_rows, cudaStream_t st) {
    if (n == 1) return launch_tail_n<1>(H, P, splits, 1, tails, gA_rows, st);
    for (int l = 0; l < n; l += kLayerBatch)
        launch_tail_n<kLayerBatch>(H, P, splits, std::min(kLayerBatch, n - l), tails + l, gA_rows, st);
}

}  // namespace ssm
