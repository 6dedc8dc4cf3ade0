// Internal launcher interface between the C-ABI layer (api.cu) and the kernel files.
#pragma once

#include "common.cuh"

namespace ssm {

// discretize.cu
void launch_discretize(int H, int P, const float2* Lambda, const float* Delta, const float2* Bc, float2* Abar,
                       float2* Bbar, cudaStream_t st);
void launch_discretize_bwd(int H, int P, const float2* Lambda, const float* Delta, const float2* Bc,
                           const float2* gAbar, const float2* gBbar, float2* dLambda, float* dDelta, float2* dB,
                           cudaStream_t st);
// Discretisation and the packed projection operands of layers in one kernel (layouts at pack_params_kernel).
// Alo: Abar's rounding residual, exp(Lambda Delta) - Abar, as fp32.  hdr (may be NULL): status word cleared.
struct PackJob {
    const float2* Lambda; const float* Delta; const float2 *Bc, *Cc;
    float2 *Abar, *Alo;
    float* Apow;   // tensor-core path with a group: powers of Abar for the kernels that scan in their epilogue
    void *WB, *WC, *Cp, *Bq;
};
// Apow: Abar^16 (a row group of those kernels), then Abar^128 (a tile), evaluated in double and rounded once; four floats
// per two neighbouring states: re, re, im, im.
constexpr int apow_floats(int P) { return 4 * P; }
constexpr int kLayerBatch = 16;   // layers of a stack that one launch of the parameter kernels takes
// Tensor-core path: WB / WC hi/lo stacked [4P, H]; group: 0 = rows in the plain order (2p + c, stacked per 128 rows:
// GemmTcTN with split_w), or the states per chain (64, 32) of the kernels that scan in their epilogue.
void launch_discretize_pack_tc(int H, int P, int group, const PackJob& job, WsHeader* hdr, cudaStream_t st);
// Plane path: the four operands as three bf16 planes: WB, WC [2P, 3H]; Cp, Bq [H, 3 * 2P].
void launch_discretize_pack_planes(int H, int P, int n, const PackJob* jobs, WsHeader* hdr, cudaStream_t st);
// CUDA-core path: fp32, WB, WC [2P, H]; Cp, Bq [H, 2P].
void launch_discretize_pack_f32(int H, int P, int n, const PackJob* jobs, WsHeader* hdr, cudaStream_t st);
// End of the backward pass of n layers of one shape.  The split-K partials [splits, H, 2P] of gBbar and dC are added;
// gBbar leaves as dB and as gamma_part_rows(H) rows of partial sums of g_gamma (gg).  Then the adjoint of the
// discretisation from rows of partial sums of gAbar [gA_rows, P] and g_gamma; sums[0] = dD and, in a stack, sums[1],
// sums[2] (LayerNorm weight and bias) from rows of partial sums [sum_rows, H].  All in a fixed order.
struct GradTail {
    const float2* Lambda; const float* Delta; const float2* Bc;
    const float *part_b, *part_c;
    float2 *dB, *dC, *gg;
    const float2* gA_part;
    float2* dLambda; float* dDelta;
    const float* sum_part[3]; int sum_rows[3]; float* sum_out[3];
};
int gamma_part_rows(int H);
void launch_layer_tail(int H, int P, int splits, int n, const GradTail* tails, int gA_rows, cudaStream_t st);

// layer_small.cu: the passes of a layer of few and narrow sequences, on the CUDA cores, a cluster of CTAs per sequence.
struct LayerSmall {
    int B, T, H, P;
    bool bf16;                // u, gy, out
    const float2* Lambda; const float* Delta; const float2 *Bc, *Cc;
    const float* D;
    const void* u;
    const uint8_t* done;      // [B, T] or NULL
    const float2 *x0, *gxT;   // [B, P] or NULL; gxT: backward
    const void* gy;           // backward
    float2* x;                // [B, T, P]: written by the forward pass, read by the backward pass
    void* out;                // y, or du
    float2 *xT, *gx0;         // [B, P] or NULL
    WsHeader* hdr;
};
int layer_small_cluster(int B, int T, int H, int P, bool bf16);   // CTAs per sequence; 0: not taken
int launch_layer_small_fwd(const LayerSmall& g, cudaStream_t st);   // also clears the status word
// B = 1: all gradients of `tail` are final.  Else gA_part [B, P] and dD_part [B, H] hold the rows of partial sums for
// launch_layer_tail, and part_b and part_c B slices, or with s (not NULL) the gradients of the states [B, T, P] are there instead.
int launch_layer_small_bwd(const LayerSmall& g, const GradTail& tail, float2* s, float2* gA_part, float* dD_part, cudaStream_t st);

// scan.cu
// Scratch the scans need for a [B,T,P] problem: a work counter and the partial sums of gAbar.
size_t scan_scratch_bytes(int B, int T, int P, int rows_per_seq = 1);   // rows_per_seq = 2: room for launch_gemm_scan_bwd_part
// Alo (may be NULL): low part of Abar, so that Abar + Alo carries the multiplier to ~48 bits.
int launch_scan_fwd(int B, int T, int P, const float2* Abar, const float2* Alo, const float2* Bu, const uint8_t* done,
                    const float2* x0, void* x, bool x_bf16, float2* xT, WsHeader* hdr, cudaStream_t st);
// x and gBu are stored both as fp32 pairs or both as bf16 pairs (x_bf16 == s_bf16).
// With gA_part / gA_rows (both or neither) the sum over the sequences is left to the caller: *gA_part points
// at *gA_rows <= kMaxPartialRows rows of P partial sums inside `scratch`, and gAbar is not written.
constexpr int kMaxPartialRows = 512;
int launch_scan_bwd(int B, int T, int P, const float2* Abar, const float2* Alo, const uint8_t* done, const float2* x0,
                    const void* x, bool x_bf16, const float2* gx, const float2* gxT, void* gBu, bool s_bf16,
                    float2* gAbar, float2* gx0, WsHeader* hdr, void* scratch, cudaStream_t st,
                    const float2** gA_part = nullptr, int* gA_rows = nullptr);

// Where a kernel that scans leaves B rows of P partial gAbar sums in `scratch`, and those brought down to *rows <= kMaxPartialRows.
float2* scan_partials(void* scratch);
const float2* reduce_scan_partials(int B, int P, void* scratch, int* rows, cudaStream_t st);

// scan_stream.cu: the scans as TMA-fed streaming kernels (a CTA walks whole sequences; all
// parallelism over time is inside the CTA).  `ticket`: one int of scratch.  The backward pass
// leaves B rows of P partial gAbar sums in `part`.
bool scan_stream_supported(int B, int T, int P);
int launch_scan_fwd_stream(int B, int T, int P, const float2* Abar, const float2* Alo, const float2* Bu,
                           const uint8_t* done, const float2* x0, void* x, bool x_bf16, float2* xT, WsHeader* hdr,
                           cudaStream_t st);
int launch_scan_bwd_stream(int B, int T, int P, const float2* Abar, const float2* Alo, const uint8_t* done,
                           const float2* x0, const void* x, bool x_bf16, const float2* gx, const float2* gxT,
                           void* gBu, float2* gx0, float2* part, WsHeader* hdr, int* ticket, cudaStream_t st);

// reduce.cu
// out[c] = sum_r in[r, c]; `tmp` must hold colsum_tmp_floats(R, C) floats.  Deterministic.
void launch_colsum(const float* in, int R, int C, float* out, float* tmp, cudaStream_t st);
size_t colsum_tmp_floats(int R, int C);
// Reduces [R, C] partial sums to at most `limit` rows (groups of rows summed in a fixed order; `in` and `tmp`,
// colsum_tmp_floats(R, C) floats, are both overwritten); returns where the rows are, *rows_out how many.
const float* launch_reduce_rows(float* in, int R, int C, float* tmp, int limit, int* rows_out, cudaStream_t st);
// part[g, c] = sum over the rows m of group g of a[m,c]*b[m,c]; a and b each fp32 or bf16.
constexpr int kDotRows = 128;
inline int dot_groups(int M) { return (M + kDotRows - 1) / kDotRows; }
size_t dot_columns_tmp_floats(int M, int C);
// The group sums only: tmp[g, c] for g < the returned number of groups.
int launch_dot_columns_partial(bool a_bf16, const void* a, bool b_bf16, const void* b, int M, int C, float* tmp,
                               cudaStream_t st);

// gemm_simt.cu: fp32-accumulate CUDA-core GEMMs (exact enough for the fp32 workloads and the
// fallback for shapes the tensor-core path does not take).
enum class Epi { StoreF32, AddDiagIo };
struct GemmTN {
    // out[m, n] = sum_k A[m, k] * Bm[n, k]   (+ diag[n] * skip[m, n] (+ add[m, n]) for AddDiagIo)
    const void* A; bool a_bf16; int lda;
    const void* Bm; bool b_bf16; int ldb;
    int M, N, K;
    Epi epi;
    void* out; bool out_bf16;            // StoreF32 ignores out_bf16
    const float* diag; const void* skip; bool skip_bf16;
    const float* add;                    // optional, fp32 [M, N]
};
void launch_gemm_tn(const GemmTN& g, cudaStream_t st);

struct GemmNT {
    // part[s, i, j] = sum_{k in slice s} A[k, i] * Bm[k, j]
    const void* A; bool a_bf16; int I;
    const float* Bm; int J;
    int K; int splits;
    float* part;
};
// part[g, c] = sum over the rows k of group g (kDotRows rows) of a[k, c] * b[k, c]: rides along with the products, on
// their K and I.
struct SimtDot {
    const void *a, *b;
    bool a_bf16, b_bf16;
    float* part;   // [dot_groups(K), I]
};
int gemm_nt_splits(int K, int I, int J);
// n = 1 or 2 products of one shape in one launch, and dot (may be NULL).
void launch_gemm_nt(const GemmNT* g, int n, const SimtDot* dot, cudaStream_t st, bool short_chains = false);

// gemm_tc.cu: bf16 projections on tcgen05 tensor cores (operands by TMA, accumulators in TMEM).
// Scan of a projection's result in its epilogue (gemm_tc_small.cu): forward, out = x with x_t = keep_t Abar x_{t-1} + acc_t, or with
// gA_part backward, out = s with s_t = acc_t + c_t, c_{t-1} = keep_t conj(Abar) s_t (c_{T-1} = gxT).
struct TileScan {
    int B, T;
    const float2 *Abar, *Alo;
    const uint8_t* done;      // [B, T] or NULL
    const float2 *x0, *gxT;   // [B, P] or NULL
    float2 *xT, *gx0;         // [B, P] or NULL
    const float2* x;          // backward: [B, T, P]
    float2* gA_part;          // backward: [B, P], sums of keep_t s_t conj(x_{t-1})
};
// Whether such a projection takes no longer than one without and a scan of its own: few tiles, whole sequences in each.
bool tc_tile_scan_supported(int B, int T, int H, int P, bool a_bf16);
struct GemmTcTN {
    // out[m, n] = sum_k A[m, k] * W[n, k];  A bf16 [M, K];  W bf16 packed by pack_params_kernel:
    // [N_out, K], or with split_w [2 * N_out, K] where each group of 256 rows holds the high
    // halves of 128 output columns followed by their low halves.
    const void* A; const void* W;
    int M, N_out, K;
    bool split_w;
    bool store_f32;                      // true: out fp32 [M, N_out]; false: out bf16 with the epilogue below
    void* out;
    const float* diag; const void* skip;   // bf16 result: out = acc + diag[n] * skip[m, n]
    WsHeader* hdr;
    // Gate (with store_f32, skip and a product schedule): besides the fp32 result also gate_out[m, n] =
    // bf16(skip[m, n] * sigmoid(acc)).
    void* gate_out = nullptr;
    // Column sums (with diag and skip): dot_part[c, n] = sum over the
    // rows m that CTA c drained of skip[m, n] * dot[m, n]; *dot_rows receives the number of rows c written
    // (at most tc_tn_dot_max_rows()).  dot: bf16 [M, N_out].
    const void* dot = nullptr;
    float* dot_part = nullptr;
    int* dot_rows = nullptr;
    // Sum of n_products products in one accumulator (fp32-accurate results from bf16 tensor-core products):
    // A is planes_a bf16 planes of K columns side by side ([M, planes_a * K]), W likewise ([N_out, planes_w * K]);
    // product j multiplies plane (prod_a >> 4 j) & 15 of A by plane (prod_w >> 4 j) & 15 of W.  fp32 result only.
    int n_products = 0, planes_a = 1, planes_w = 1;
    uint32_t prod_a = 0, prod_w = 0;
    // (These are left to the kernel of gemm_tc_small.cu; skip, dot and add in any type also to gemm_tc_planes.cu.)
    bool a_f32 = false;                  // A is fp32 [M, K]; its three planes are made on the way to the tensor cores ...
    void* a_planes_out = nullptr;        // ... and, if asked for, stored [M, 3K] for a later kernel
    bool skip_bf16 = true, dot_bf16 = true;   // types of skip and dot; with diag and store_f32 the result is fp32
    const float* add = nullptr;          // fp32 [M, N_out], added to acc + diag * skip
    const TileScan* scan = nullptr;
};
bool tc_tn_supported(int M, int N_out, int K, bool split_w);
int launch_gemm_tc_tn_small(const GemmTcTN& g, cudaStream_t st);
bool tc_planes_many_tiles(int M, int N_out);
int launch_gemm_tc_planes(const GemmTcTN& g, cudaStream_t st);   // gemm_tc_planes.cu: products of planes, many tiles
int tc_tn_small_max_dot_rows(int M);
int tc_max_n();   // widest output of the tensor-core projections
bool tc_tn_dot_supported(int M, int N_out);
int tc_tn_dot_max_rows(int M);
int launch_gemm_tc_tn(const GemmTcTN& g, cudaStream_t st);

// One step for B trajectories in one kernel (gemm_tc_step.cu), from the operands of the tensor-core path (f32 = false:
// Wb hi/lo stacked [4P, H] in the plain order, Wc [H, 2P]) or of the plane path (f32: Wb [2P, 3H], Wc [H, 6P]).
struct StepCall {
    int B, H, P;
    bool f32;
    const void *Wb, *Wc;
    const float2 *Abar, *Alo;
    const float* D;
    const void* u;             // [B, H] io
    const uint8_t* done;       // [B] or NULL
    const float2* x_prev;      // [B, P]
    float2* x_next;            // [B, P]; may be x_prev
    void* x_bf16;              // scratch [B, 2P] bf16 (f32: unused)
    void* y;                   // [B, H] io
    WsHeader* hdr;
};
bool use_step_kernel(int H, int P, bool f32);
int launch_step(const StepCall& g, cudaStream_t st);
// The same for a few trajectories, on the CUDA cores (step_small.cu).
bool use_step_small(int B, int H, int P);
int launch_step_small(const StepCall& g, cudaStream_t st);

// Input projection and forward scan fused (gemm_tc.cu): x = scan(u Bbar^T) written as the two bf16
// planes of x; Bu never reaches memory.  For lengths that fill most of their 128-row tiles (or 16, 32, 64: a
// tile then holds whole sequences) and enough (sequence, 64 states) chains (tc_gemm_scan_fwd_supported).
struct GemmScanFwd {
    const void* u;          // bf16 [B*T, H]
    const void* Wsplit;     // hi/lo stacked Bbar operand [4P, H] (as for GemmTcTN with split_w)
    int B, T, H, P;
    const float2* Abar;     // [P]
    const float* Apow;      // powers of Abar (PackJob)
    const uint8_t* done;    // [B*T] or NULL
    const float2* x0;       // [B, P] or NULL
    void* x_planes;         // out: bf16 hi plane [B*T, 2P], then the lo plane
    float2* xT;             // out [B, P] or NULL
    WsHeader* hdr;
};
bool tc_gemm_scan_fwd_supported(int B, int T, int H, int P);
// States per chain these kernels (forward and backward alike) use for a problem: 64 or 32; 0: not taken.  The
// hi/lo stacked operands they read are packed for that group size (launch_discretize_pack_tc).
int tc_gemm_scan_group(int B, int T, int H, int P);
// Whether these kernels put both CTAs of a pair on one sequence for a problem (few long sequences).
bool tc_gemm_scan_time_pairs(int B, int T, int H, int P);
int launch_gemm_scan_fwd(const GemmScanFwd& g, cudaStream_t st);

// g_x projection and reverse scan fused (gemm_tc.cu): s = reverse scan(gy conj(C)) written as the two
// bf16 planes of s, the sums s_t conj(x_{t-1}) per (sequence, state) in gA_part; g_x never reaches
// memory.  Lengths and chains as for the forward kernel (tc_gemm_scan_bwd_supported).
struct GemmScanBwd {
    const void* gy;         // bf16 [B*T, H]
    const void* Wsplit;     // hi/lo stacked conj(C) operand [4P, H], rows in the pair_cols order
    int B, T, H, P;
    const float2* Abar;     // [P]
    const float* Apow;      // powers of Abar (PackJob)
    const uint8_t* done;    // [B*T] or NULL
    const float2* x0;       // [B, P] or NULL
    const float2* gxT;      // [B, P] or NULL
    const void* x_planes;   // bf16 hi plane [B*T, 2P], then the lo plane
    void* s_planes;         // out: the same layout
    float2* gA_part;        // out [tc_gemm_scan_bwd_part_rows(B, T, H, P), P]
    float2* gx0;            // out [B, P] or NULL
    WsHeader* hdr;
};
bool tc_gemm_scan_bwd_supported(int B, int T, int H, int P);
int tc_gemm_scan_bwd_part_rows(int B, int T, int H, int P);   // rows of gA_part the kernel writes (at most 2 B)
int launch_gemm_scan_bwd(const GemmScanBwd& g, cudaStream_t st);
// scan.cu: the same with gA_part placed in `scratch` (as for launch_scan_bwd) and brought down to
// *gA_rows <= kMaxPartialRows rows at *gA_part_out; the caller sums those.
int launch_gemm_scan_bwd_part(GemmScanBwd g, void* scratch, const float2** gA_part_out, int* gA_rows, cudaStream_t st);

// Weight-gradient products: part[s, i, j] = sum_{m in slice s} A[m, i] * (Bm_hi[m, j] + Bm_lo[m, j]);  A bf16 [K, I]
// with lda elements between rows, Bm_hi / Bm_lo bf16 [K, J]: the two planes of a state tensor.
struct GemmTcNT {
    const void* A; int lda;
    const void* Bm_hi; const void* Bm_lo;
    float* part;   // [splits, I, J]
};
bool tc_nt_supported(int I, int J);
// Slices of the rows for a pair of products of one shape.
int tc_nt_splits(int K, int I, int J);
int launch_gemm_tc_nt2(int K, int I, int J, int splits, const GemmTcNT& g0, const GemmTcNT& g1, WsHeader* hdr, cudaStream_t st);
// Weight-gradient products of fp32 layers from planes (gemm_tc_nt_planes.cu), two per layer: A = planes_a planes of I
// columns side by side, B = planes_b planes of J columns; product schedules as in GemmTcTN.  I, J multiples of 128.
struct GemmTcNtPlanes {
    const void *A, *B;
    int planes_a, planes_b, n_products;
    uint32_t prod_a, prod_b;
    float* part;   // [splits, I, J]
};
int tc_nt_planes_splits(int K, int I, int J, int n_products);
int launch_gemm_tc_nt_planes(int K, int I, int J, int splits, int n_products, const GemmTcNtPlanes* products, WsHeader* hdr,
                             cudaStream_t st);

// planes.cu: fp32 tensors as three bf16 planes side by side ([M, K] -> [M, 3K]).
void launch_split_planes(const float* in, size_t M, int K, void* out, cudaStream_t st);

// glu.cu: what surrounds the GEMMs of the half-GLU gate out = v * sigmoid(GELU(v) W).
// Tensor-core path (may be NULL): Wz, Wn [H, 2H], hi | lo planes of W transposed (z = x1 W) and of W (g_x1 = gz W^T);
// Wt_f32 (CUDA-core path, may be NULL): W transposed.  Clears the header's status word.
// x1 = GELU(v) in the same launch; planes: bf16 [M, 2H], high halves in columns [0, H), low halves in [H, 2H); else fp32 [M, H]
void launch_glu_pre(bool io_bf16, bool planes, size_t n, int H, const void* v, void* x1, const float* W, void* Wz, void* Wn,
                    float* Wt_f32, WsHeader* hdr, cudaStream_t st);
void launch_glu_out(bool io_bf16, size_t n, const void* v, const float* z, void* out, cudaStream_t st);
// gz = gout * v * s (1 - s), s = sigmoid(z); planes: two bf16 planes (hi, lo) n elements apart, else fp32
void launch_glu_gz(bool io_bf16, bool planes, size_t n, const void* v, const void* gout, const float* z, void* gz,
                   cudaStream_t st);
// dW = the sum of `splits` slices of n_w elements, and gv = gout * sigmoid(z) + g_x1 * GELU'(v)
void launch_glu_post(bool io_bf16, const float* part, int splits, size_t n_w, float* dW, size_t n, const void* v, const void* gout,
                     const float* z, const float* gx1, void* gv, cudaStream_t st);

// stack.cu: out = LayerNorm(u + GELU(v)) * w + b per row of H features, and its backward
// (gz = LN'(g), gv = gz * GELU'(v), dw, db).  v, gz, gv are fp32; u, out and g are fp32 or bf16 as
// flagged (only the stack's own input, output and output gradient are in the I/O type).
// tmp: stack_tmp_floats(M, H) floats.
size_t stack_tmp_floats(int M, int H);
void launch_stack_fwd(bool u_bf16, bool out_bf16, int M, int H, const void* u, const float* v, const float* w,
                      const float* b, void* out, float* mu, float* rstd, cudaStream_t st);
// The sums for dw and db are left as *part_rows <= kMaxPartialRows rows of [H] each, inside tmp.
void launch_stack_bwd(bool g_bf16, bool u_bf16, int M, int H, const void* g, const void* u, const float* v,
                      const float* w, const float* mu, const float* rstd, float* gz, float* gv, float* tmp,
                      const float** dw_part, const float** db_part, int* part_rows, cudaStream_t st);

}  // namespace ssm
