// C-ABI entry points (see include/ssm.h): argument checks, workspace layout, launch order.
#include <cstdio>
#include <algorithm>

#include "kernels.h"

using namespace ssm;

#define SSM_API extern "C" __attribute__((visibility("default")))

namespace {

// Workspace of one layer.  Two paths:
//  * tensor-core path (bf16 I/O and tile-sized H, P): projections on tcgen05, states Bu / g_x
//    in one fp32 buffer, x and s kept as bf16 pairs;
//  * CUDA-core path (fp32 I/O, or odd shapes): fp32 weights and states throughout.
//  * plane path (fp32 I/O and tile-sized H, P with enough rows): the same projections on tcgen05 as sums
//    of products of bf16 planes (three planes per fp32 value: exact), fp32 states, scans as on the
//    CUDA-core path.
//  * small layers off the tensor cores: each pass in one kernel, a cluster per sequence; fp32 x is all that is kept.
struct LayerPlan {
    bool tc;
    bool planes;
    bool small, slices;   // slices: of the weight gradients, by the small layer's kernel
    int splits;
    size_t hdr, Abar, Alo, Apow, W0, W1, W2, W3, f32buf, xs, gs, gAbar, gg, scan, part, dot, total;
    size_t u3, gy3, x3, s3;   // plane path: planes of u, gy, x, s for the weight gradients
};

// fp32 layers of tile-sized widths.  us per forward and backward pass, CUDA cores / planes, at H, P = 384, 192: 50 rows
// 106 / 61, 1024 rows 132 / 74, 40000 rows 2355 / 541; at 128, 64: 8 rows 49 / 53, 64 rows 52 / 53, 1024 rows 58 / 57, 30000
// rows 274 / 174.  Errors against float64 are smaller with planes: 40000 rows at 384, 192: y 1.6e-7 / 1.2e-7, du 8.8e-8 / 6.9e-8 in
// the 2-norm, the gradient sums by as much or more.
// Single steps take them at every batch size: the operands prepared for one are read at any other (us per step in a graph, fp32
// weights on the CUDA cores / planes, 8 trajectories: 384, 192 39.4 / 7.1; 128, 64 15.1 / 3.5).
bool planes_supported(const ssm_shape& s, bool step) {
    const double work = (double)s.B * s.T * s.H * 2 * s.P;
    return s.H % 128 == 0 && s.P % 64 == 0 && s.H <= tc_max_n() && 2 * s.P <= tc_max_n() &&
           (step || work >= (1 << 21) || (s.H % 256 == 0 && s.P % 128 == 0));
}
// Product schedules (plane of the first operand, plane of the second, four bits each, smallest terms first):
// fp32 x fp32 = lo hi, hi lo, mid mid, mid hi, hi mid, hi hi;  bf16 x fp32 = hi lo, hi mid, hi hi.
constexpr uint32_t kProd6A = 0x001102u, kProd6B = 0x010120u;
constexpr uint32_t kProd3A = 0x000u, kProd3B = 0x012u;

constexpr int kMaxStackLayers = 64;

size_t take(size_t& off, size_t bytes) {
    const size_t at = off;
    off = align_up(off + bytes, 256);
    return at;
}

// step: the workspace of single-step mode (T = 1), whose path and layout up to the packed operands go by the widths alone.
LayerPlan plan_layer(const ssm_shape& s, bool allow_tc = true, bool step = false) {
    LayerPlan p{};
    size_t off = 0;
    const size_t BT = (size_t)s.B * s.T, PH = (size_t)s.P * s.H;
    const int P2 = 2 * s.P;
    p.tc = allow_tc && s.io_dtype == SSM_BF16 && tc_tn_supported((int)BT, P2, s.H, true) &&
           tc_tn_supported((int)BT, s.H, P2, false) && tc_nt_supported(s.H, P2);
    p.planes = !p.tc && s.io_dtype == SSM_F32 && planes_supported(s, step);
    p.splits = p.tc ? tc_nt_splits((int)BT, s.H, P2) : (p.planes ? tc_nt_planes_splits((int)BT, s.H, P2, 2) : gemm_nt_splits((int)BT, s.H, P2));
    p.hdr = take(off, sizeof(WsHeader));
    p.Abar = take(off, (size_t)s.P * 8);
    p.Alo = take(off, (size_t)s.P * 8);
    if (p.tc) {
        p.Apow = take(off, (size_t)apow_floats(s.P) * 4);
        p.W0 = take(off, 4 * PH * 2);   // hi/lo stacked Bbar operand  [4P, H] bf16
        p.W1 = take(off, 4 * PH * 2);   // hi/lo stacked conj(C) operand [4P, H] bf16
        p.W2 = take(off, 2 * PH * 2);   // Cp [H, 2P] bf16
        p.W3 = take(off, 2 * PH * 2);   // Bq [H, 2P] bf16
        p.f32buf = take(off, BT * s.P * 8);   // Bu (forward), then g_x (backward)
        p.xs = take(off, BT * s.P * 8);       // x as two bf16 planes (hi, lo)
        p.gs = take(off, BT * s.P * 8);       // s as two bf16 planes (hi, lo)
    } else {
        // CUDA-core path: fp32 operands.  Plane path: three bf16 planes of each (6 PH values, 2 bytes each).
        p.W0 = take(off, p.planes ? 6 * PH * 2 : 2 * PH * 4);   // Bp [2P, H]   | Wb3 [2P, 3H]
        p.W1 = take(off, p.planes ? 6 * PH * 2 : 2 * PH * 4);   // Cq [2P, H]   | Cq3 [2P, 3H]
        p.W2 = take(off, p.planes ? 6 * PH * 2 : 2 * PH * 4);   // Cp [H, 2P]   | Cp3 [H, 3 * 2P]
        p.W3 = take(off, p.planes ? 6 * PH * 2 : 2 * PH * 4);   // Bq [H, 2P]   | Bq3 [H, 3 * 2P]
        p.f32buf = off;                 // unused
        p.xs = take(off, BT * s.P * 8); // Bu, overwritten in place by x
        p.gs = take(off, BT * s.P * 8); // g_x, overwritten in place by s
        if (p.planes) {
            p.u3 = take(off, BT * 3 * s.H * 2);
            p.gy3 = take(off, BT * 3 * s.H * 2);
            p.x3 = take(off, BT * 6 * s.P * 2);
            p.s3 = take(off, BT * 6 * s.P * 2);
        }
    }
    p.gAbar = take(off, (size_t)s.P * 8);
    p.gg = take(off, (size_t)gamma_part_rows(s.H) * s.P * 8);
    p.scan = take(off, scan_scratch_bytes(s.B, s.T, s.P, 2));
    p.part = take(off, (size_t)2 * p.splits * 2 * PH * 4);   // split-K partials of gBbar, then those of dC
    {   // dD: partial column sums of gy * u, from the stand-alone kernel or from the epilogue of the du projection
        const size_t rows = (size_t)tc_tn_dot_max_rows((int)BT);
        const size_t fused = rows * s.H + colsum_tmp_floats((int)rows, s.H);
        p.dot = take(off, std::max(dot_columns_tmp_floats((int)BT, s.H), fused) * 4);
    }
    p.total = off;
    if (allow_tc && !step && !p.tc && !p.planes && layer_small_cluster(s.B, s.T, s.H, s.P, s.io_dtype == SSM_BF16) > 0) {
        // The passes in one kernel keep x, and with several sequences a slice of both weight gradients for each of them where that
        // fits what the separate kernels need, so that no batch needs more than a larger one (32 x 10 (184, 128) would want
        // 13.8 MB, 33 x 10 and the separate kernels 4.0).  Otherwise s, which the separate kernels' products take.
        LayerPlan q{};
        for (const bool slices : {true, false}) {
            off = 0;
            q.small = true;
            q.slices = slices;
            q.splits = slices ? s.B : p.splits;
            q.hdr = take(off, sizeof(WsHeader));
            q.xs = take(off, BT * s.P * 8);
            q.gs = take(off, slices ? 0 : BT * s.P * 8);
            q.gg = take(off, (size_t)gamma_part_rows(s.H) * s.P * 8);
            q.scan = take(off, (size_t)s.B * s.P * 8);   // gAbar of every sequence
            q.dot = take(off, (size_t)s.B * s.H * 4);
            q.part = take(off, s.B > 1 ? (size_t)2 * q.splits * 2 * PH * 4 : 0);
            q.total = p.total;
            if (off <= q.total) return q;
        }
    }
    return p;
}

template <typename T>
T* at(void* ws, size_t off) { return reinterpret_cast<T*>(reinterpret_cast<char*>(ws) + off); }

int check_ws(const void* ws, size_t have, size_t need) {
    if (!ws) return SSM_ERR_WORKSPACE;
    if (misaligned(ws, 256)) return SSM_ERR_ALIGN;
    if (have < need) return SSM_ERR_WORKSPACE;
    return SSM_OK;
}

}  // namespace

SSM_API const char* ssm_status_string(int status) {
    switch (status) {
        case SSM_OK: return "ok";
        case SSM_ERR_NULL: return "a required pointer is NULL";
        case SSM_ERR_SHAPE: return "bad shape (B,T >= 1; H,P positive multiples of 8; reserved == 0)";
        case SSM_ERR_ALIGN: return "a pointer is not aligned as required";
        case SSM_ERR_DTYPE: return "io_dtype must be SSM_F32 or SSM_BF16";
        case SSM_ERR_WORKSPACE: return "workspace missing or too small";
        case SSM_ERR_CUDA: return "a CUDA call or kernel launch failed";
        case SSM_ERR_TIMEOUT: return "a bounded device-side wait gave up";
        case SSM_ERR_TOO_LARGE: return "problem needs more scratch than the library's built-in static buffer holds";
        default: return "unknown status";
    }
}

SSM_API int ssm_check(const void* ws, void* stream) {
    if (!ws) return SSM_ERR_NULL;
    int status = 0;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(&status, ws, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return SSM_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SSM_ERR_CUDA;
    return status == 0 ? SSM_OK : SSM_ERR_TIMEOUT;
}

SSM_API int ssm_discretize(const ssm_shape* shape, const ssm_c64* Lambda, const float* Delta, const ssm_c64* Bc,
                           ssm_c64* Abar, ssm_c64* Bbar, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Lambda || !Delta || !Bc || !Abar || !Bbar) return SSM_ERR_NULL;
    if (misaligned(Lambda) || misaligned(Delta) || misaligned(Bc) || misaligned(Abar) || misaligned(Bbar))
        return SSM_ERR_ALIGN;
    launch_discretize(shape->H, shape->P, (const float2*)Lambda, Delta, (const float2*)Bc, (float2*)Abar, (float2*)Bbar,
                      (cudaStream_t)stream);
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_discretize_bwd(const ssm_shape* shape, const ssm_c64* Lambda, const float* Delta,
                               const ssm_c64* Bc, const ssm_c64* gAbar, const ssm_c64* gBbar, ssm_c64* dLambda,
                               float* dDelta, ssm_c64* dB, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Lambda || !Delta || !Bc || !gAbar || !gBbar || !dLambda || !dDelta || !dB) return SSM_ERR_NULL;
    if (misaligned(Lambda) || misaligned(Delta) || misaligned(Bc) || misaligned(gAbar) || misaligned(gBbar) ||
        misaligned(dLambda) || misaligned(dDelta) || misaligned(dB))
        return SSM_ERR_ALIGN;
    launch_discretize_bwd(shape->H, shape->P, (const float2*)Lambda, Delta, (const float2*)Bc,
                          (const float2*)gAbar, (const float2*)gBbar, (float2*)dLambda, dDelta, (float2*)dB,
                          (cudaStream_t)stream);
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API size_t ssm_scan_workspace_bytes(const ssm_shape* shape) {
    if (check_shape(shape) != SSM_OK) return 0;
    return sizeof(WsHeader) + scan_scratch_bytes(shape->B, shape->T, shape->P);
}

SSM_API int ssm_scan_fwd(const ssm_shape* shape, const ssm_c64* Abar, const ssm_c64* Bu, const uint8_t* done,
                         const ssm_c64* x0, ssm_c64* x, ssm_c64* xT, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Abar || !Bu || !x) return SSM_ERR_NULL;
    if (misaligned(Abar) || misaligned(Bu) || misaligned(x) || misaligned(x0) || misaligned(xT)) return SSM_ERR_ALIGN;
    if (int rc = check_ws(ws, ws_bytes, ssm_scan_workspace_bytes(shape))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(ws, 0, sizeof(WsHeader), st) != cudaSuccess) return SSM_ERR_CUDA;
    StageTimer tm("scan_fwd", st);
    int rc = launch_scan_fwd(shape->B, shape->T, shape->P, (const float2*)Abar, nullptr, (const float2*)Bu, done,
                             (const float2*)x0, x, false, (float2*)xT, at<WsHeader>(ws, 0), st);
    if (rc) return rc;
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_scan_bwd(const ssm_shape* shape, const ssm_c64* Abar, const uint8_t* done, const ssm_c64* x0,
                         const ssm_c64* x, const ssm_c64* gx, const ssm_c64* gxT, ssm_c64* gBu, ssm_c64* gAbar,
                         ssm_c64* gx0, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Abar || !x || !gx || !gBu || !gAbar) return SSM_ERR_NULL;
    if (misaligned(Abar) || misaligned(x) || misaligned(gx) || misaligned(gBu) || misaligned(gAbar) ||
        misaligned(x0) || misaligned(gxT) || misaligned(gx0))
        return SSM_ERR_ALIGN;
    if (int rc = check_ws(ws, ws_bytes, ssm_scan_workspace_bytes(shape))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(ws, 0, sizeof(WsHeader), st) != cudaSuccess) return SSM_ERR_CUDA;
    StageTimer tm("scan_bwd", st);
    int rc = launch_scan_bwd(shape->B, shape->T, shape->P, (const float2*)Abar, nullptr, done, (const float2*)x0, x, false,
                             (const float2*)gx, (const float2*)gxT, gBu, false, (float2*)gAbar, (float2*)gx0,
                             at<WsHeader>(ws, 0), at<char>(ws, sizeof(WsHeader)), st);
    if (rc) return rc;
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API size_t ssm_layer_workspace_bytes(const ssm_shape* shape) {
    if (check_shape(shape) != SSM_OK) return 0;
    return plan_layer(*shape).total;
}

SSM_API int ssm_layer_plan_string(const ssm_shape* shape, char* buf, size_t len) {
    if (!buf || len == 0) return SSM_ERR_NULL;
    buf[0] = 0;
    if (int rc = check_shape(shape)) return rc;
    const ssm_shape& s = *shape;
    const LayerPlan p = plan_layer(s);
    const int group = p.tc ? tc_gemm_scan_group(s.B, s.T, s.H, s.P) : 0;
    const char* proj = p.tc ? "tensor-cores" : (p.planes ? "tensor-cores-planes" : "cuda-cores");
    const bool in_epilogue = p.planes && tc_tile_scan_supported(s.B, s.T, s.H, s.P, false);
    if (group)
        snprintf(buf, len, "projections=%s scans=fused chain_states=%d time_pairs=%d", proj, group,
                 tc_gemm_scan_time_pairs(s.B, s.T, s.H, s.P) ? 1 : 0);
    else
        snprintf(buf, len, "projections=%s scans=%s", proj, p.small ? "one-kernel" : in_epilogue ? "in-epilogue" : "separate");
    return SSM_OK;
}

// Discretised parameters and packed projection operands into the workspace; clears the status word of `hdr` if given.
static PackJob pack_job(const LayerPlan& p, const ssm_c64* Lambda, const float* Delta, const ssm_c64* Bc, const ssm_c64* Cc,
                        void* ws) {
    return {(const float2*)Lambda, Delta, (const float2*)Bc, (const float2*)Cc, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo),
            at<float>(ws, p.Apow), at<void>(ws, p.W0), at<void>(ws, p.W1), at<void>(ws, p.W2), at<void>(ws, p.W3)};
}
static void layer_prepare(const ssm_shape& s, const LayerPlan& p, const ssm_c64* Lambda, const float* Delta,
                          const ssm_c64* Bc, const ssm_c64* Cc, void* ws, WsHeader* hdr, cudaStream_t st) {
    StageTimer tm("discretize_pack", st);
    const PackJob job = pack_job(p, Lambda, Delta, Bc, Cc, ws);
    if (p.tc)   // (the kernels that scan in the epilogue of a projection want their own column order)
        launch_discretize_pack_tc(s.H, s.P, tc_gemm_scan_group(s.B, s.T, s.H, s.P), job, hdr, st);
    else if (p.planes)
        launch_discretize_pack_planes(s.H, s.P, 1, &job, hdr, st);
    else
        launch_discretize_pack_f32(s.H, s.P, 1, &job, hdr, st);
}

// One projection of the plane path.  `g` has its fp32 or bf16 operand in A; `planes` is where the planes of an fp32
// operand go (keep: they are wanted later, by the weight gradients).
static int plane_projection(GemmTcTN g, bool a_bf16, void* planes, bool keep, cudaStream_t st) {
    g.n_products = a_bf16 ? 3 : 6;
    g.planes_a = a_bf16 ? 1 : 3;
    g.planes_w = 3;
    g.prod_a = a_bf16 ? kProd3A : kProd6A;
    g.prod_w = a_bf16 ? kProd3B : kProd6B;
    if (tc_planes_many_tiles(g.M, g.N_out)) {
        if (!a_bf16) {
            launch_split_planes((const float*)g.A, (size_t)g.M, g.K, planes, st);
            g.A = planes;
        }
        return launch_gemm_tc_planes(g, st);
    }
    if (!a_bf16) g.a_f32 = true, g.a_planes_out = keep ? planes : nullptr;
    return launch_gemm_tc_tn(g, st);
}

// Launch sequence of one layer's forward pass from a prepared workspace.  `hdr` receives the
// status of bounded waits.  keep_planes: a backward pass will follow (fp32 layers leave the planes of u and x for it).
// Storage types of the tensors a layer reads and writes.  For the entry points of a single layer all
// of them are shape->io_dtype; inside a stack only the stack's own input and outputs are.
struct LayerIo {
    bool u_bf16, y_bf16;      // forward: u in, y out
    bool gy_bf16, du_bf16;    // backward: gy in, du out
};
static LayerIo layer_io(const ssm_shape& s) {
    const bool b = s.io_dtype == SSM_BF16;
    return {b, b, b, b};
}

static int layer_fwd_run(const ssm_shape& s, const LayerPlan& p, const LayerIo& io, const float* D, const void* u,
                         const uint8_t* done, const ssm_c64* x0, void* y, ssm_c64* xT, void* ws, WsHeader* hdr,
                         bool keep_planes, cudaStream_t st) {
    const int BT = s.B * s.T, P2 = 2 * s.P;
    if (p.tc && !(io.u_bf16 && io.y_bf16)) return SSM_ERR_DTYPE;   // the tensor-core path reads and writes bf16
    int rc = SSM_OK;
    if (p.tc && tc_gemm_scan_fwd_supported(s.B, s.T, s.H, s.P)) {
        {   // projection and scan in one kernel: x = scan(u Bbar^T), Bu stays on chip
            StageTimer tm("gemm_Bu_scan_fwd", st);
            GemmScanFwd g{u, at<void>(ws, p.W0), s.B, s.T, s.H, s.P, at<float2>(ws, p.Abar), at<float>(ws, p.Apow), done, (const float2*)x0,
                          at<void>(ws, p.xs), (float2*)xT, hdr};
            if ((rc = launch_gemm_scan_fwd(g, st))) return rc;
        }
        {   // y[m,h] = sum_k x[m,k] Cp[h,k] + D[h] u[m,h]
            StageTimer tm("gemm_y", st);
            GemmTcTN g{at<void>(ws, p.xs), at<void>(ws, p.W2), BT, s.H, P2, false, false, y, D, u, hdr};
            if ((rc = launch_gemm_tc_tn(g, st))) return rc;
        }
    } else if (p.tc) {
        {   // Bu[m, 2p+c] = sum_h u[m,h] Bbar_c[p,h]     (weights as hi + lo bf16)
            StageTimer tm("gemm_Bu", st);
            GemmTcTN g{u, at<void>(ws, p.W0), BT, P2, s.H, true, true, at<void>(ws, p.f32buf), nullptr, nullptr, hdr};
            if ((rc = launch_gemm_tc_tn(g, st))) return rc;
        }
        {
            StageTimer tm("scan_fwd", st);
            rc = launch_scan_fwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), at<float2>(ws, p.f32buf), done,
                                 (const float2*)x0, at<void>(ws, p.xs), true, (float2*)xT, hdr, st);
            if (rc) return rc;
        }
        {   // y[m,h] = sum_k x[m,k] Cp[h,k] + D[h] u[m,h]
            StageTimer tm("gemm_y", st);
            GemmTcTN g{at<void>(ws, p.xs), at<void>(ws, p.W2), BT, s.H, P2, false, false, y, D, u, hdr};
            if ((rc = launch_gemm_tc_tn(g, st))) return rc;
        }
    } else if (p.planes) {
        if (tc_tile_scan_supported(s.B, s.T, s.H, s.P, io.u_bf16)) {
            StageTimer tm("scan_fwd", st);   // Bu as below, scanned in the projection's epilogue
            TileScan scan{s.B, s.T, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), done, (const float2*)x0, nullptr, (float2*)xT};
            GemmTcTN g{u, at<void>(ws, p.W0), BT, P2, s.H, false, true, at<void>(ws, p.xs), nullptr, nullptr, hdr};
            g.scan = &scan;
            if ((rc = plane_projection(g, io.u_bf16, at<void>(ws, p.u3), keep_planes, st))) return rc;
        } else {
        {   // Bu = u Bbar^T as a sum of plane products (u: three planes of an fp32 input, or the bf16 input itself)
            StageTimer tm("gemm_Bu", st);
            const GemmTcTN g{u, at<void>(ws, p.W0), BT, P2, s.H, false, true, at<void>(ws, p.xs), nullptr, nullptr, hdr};
            if ((rc = plane_projection(g, io.u_bf16, at<void>(ws, p.u3), keep_planes, st))) return rc;
        }
        {
            StageTimer tm("scan_fwd", st);
            rc = launch_scan_fwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), at<float2>(ws, p.xs), done,
                                 (const float2*)x0, at<void>(ws, p.xs), false, (float2*)xT, hdr, st);
            if (rc) return rc;
        }
        }
        {   // y = x Cp^T + D u: six products of planes, the skip term in the epilogue
            StageTimer tm("gemm_y", st);
            GemmTcTN g{at<void>(ws, p.xs), at<void>(ws, p.W2), BT, s.H, P2, false, !io.y_bf16, y, D, u, hdr};
            g.skip_bf16 = io.u_bf16;
            if ((rc = plane_projection(g, false, at<void>(ws, p.x3), keep_planes, st))) return rc;
        }
    } else {
        {
            StageTimer tm("gemm_Bu", st);
            GemmTN g1{u, io.u_bf16, s.H, at<void>(ws, p.W0), false, s.H, BT, P2, s.H, Epi::StoreF32,
                      at<void>(ws, p.xs), false, nullptr, nullptr, false, nullptr};
            launch_gemm_tn(g1, st);
        }
        {
            StageTimer tm("scan_fwd", st);
            rc = launch_scan_fwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), at<float2>(ws, p.xs), done,
                                 (const float2*)x0, at<void>(ws, p.xs), false, (float2*)xT, hdr, st);
            if (rc) return rc;
        }
        {
            StageTimer tm("gemm_y", st);
            GemmTN g2{at<void>(ws, p.xs), false, P2, at<void>(ws, p.W2), false, P2, BT, s.H, P2, Epi::AddDiagIo,
                      y, io.y_bf16, D, u, io.u_bf16, nullptr};
            launch_gemm_tn(g2, st);
        }
    }
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

static int layer_fwd_impl(const ssm_shape& s, const LayerPlan& p, const LayerIo& io, const ssm_c64* Lambda,
                          const float* Delta, const ssm_c64* Bc, const ssm_c64* Cc, const float* D, const void* u,
                          const uint8_t* done, const ssm_c64* x0, void* y, ssm_c64* xT, void* ws, WsHeader* hdr,
                          cudaStream_t st) {
    layer_prepare(s, p, Lambda, Delta, Bc, Cc, ws, hdr, st);
    return layer_fwd_run(s, p, io, D, u, done, x0, y, xT, ws, hdr, true, st);
}

SSM_API int ssm_layer_fwd(const ssm_shape* shape, const ssm_c64* Lambda, const float* Delta, const ssm_c64* Bc,
                          const ssm_c64* Cc, const float* D, const void* u, const uint8_t* done,
                          const ssm_c64* x0, void* y, ssm_c64* xT, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Lambda || !Delta || !Bc || !Cc || !D || !u || !y) return SSM_ERR_NULL;
    if (misaligned(Lambda) || misaligned(Delta) || misaligned(Bc) || misaligned(Cc) || misaligned(D) ||
        misaligned(u) || misaligned(y) || misaligned(x0) || misaligned(xT))
        return SSM_ERR_ALIGN;
    const ssm_shape& s = *shape;
    const LayerPlan p = plan_layer(s);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    WsHeader* hdr = at<WsHeader>(ws, p.hdr);
    if (p.small) {
        StageTimer tm("scan_fwd", st);   // (with everything around the scan)
        const LayerSmall g{s.B, s.T, s.H, s.P, s.io_dtype == SSM_BF16, (const float2*)Lambda, Delta, (const float2*)Bc, (const float2*)Cc,
                           D, u, done, (const float2*)x0, nullptr, nullptr, at<float2>(ws, p.xs), y, (float2*)xT, nullptr, hdr};
        if (int rc = launch_layer_small_fwd(g, st)) return rc;
        SSM_RETURN_IF_CUDA_ERROR();
        return SSM_OK;
    }
    return layer_fwd_impl(s, p, layer_io(s), Lambda, Delta, Bc, Cc, D, u, done, x0, y, xT, ws, hdr, st);
}

// Single-step mode: the layer's forward launch sequence for T = 1 from operands prepared once.
static ssm_shape step_shape(const ssm_shape& s) {
    ssm_shape t = s;
    t.T = 1;
    return t;
}

SSM_API size_t ssm_step_workspace_bytes(const ssm_shape* shape) {
    if (check_shape(shape) != SSM_OK) return 0;
    return plan_layer(step_shape(*shape), true, true).total;
}

SSM_API int ssm_step_prepare(const ssm_shape* shape, const ssm_c64* Lambda, const float* Delta, const ssm_c64* Bc,
                             const ssm_c64* Cc, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Lambda || !Delta || !Bc || !Cc) return SSM_ERR_NULL;
    if (misaligned(Lambda) || misaligned(Delta) || misaligned(Bc) || misaligned(Cc)) return SSM_ERR_ALIGN;
    const ssm_shape s = step_shape(*shape);
    const LayerPlan p = plan_layer(s, true, true);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    layer_prepare(s, p, Lambda, Delta, Bc, Cc, ws, at<WsHeader>(ws, p.hdr), st);
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_step(const ssm_shape* shape, const float* D, const void* u, const uint8_t* done,
                     const ssm_c64* x_prev, ssm_c64* x_next, void* y, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!D || !u || !x_prev || !x_next || !y) return SSM_ERR_NULL;
    if (misaligned(D) || misaligned(u) || misaligned(x_prev) || misaligned(x_next) || misaligned(y))
        return SSM_ERR_ALIGN;
    const ssm_shape s = step_shape(*shape);
    const LayerPlan p = plan_layer(s, true, true);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    // each (trajectory, state) is read as x0 and written as xT by the same thread, so x_next may be x_prev
    const bool few = use_step_small(s.B, s.H, s.P);
    if ((p.tc || p.planes) && (few || use_step_kernel(s.H, s.P, p.planes))) {
        StageTimer tm("step", (cudaStream_t)stream);
        const StepCall g{s.B, s.H, s.P, p.planes, at<void>(ws, p.W0), at<void>(ws, p.W2), at<float2>(ws, p.Abar), at<float2>(ws, p.Alo),
                         D, u, done, (const float2*)x_prev, (float2*)x_next, at<void>(ws, p.xs), y, at<WsHeader>(ws, p.hdr)};
        const int rc = few ? launch_step_small(g, (cudaStream_t)stream) : launch_step(g, (cudaStream_t)stream);
        if (rc) return rc;
        SSM_RETURN_IF_CUDA_ERROR();
        return SSM_OK;
    }
    return layer_fwd_run(s, p, layer_io(s), D, u, done, x_prev, y, x_next, ws, at<WsHeader>(ws, p.hdr), false,
                         (cudaStream_t)stream);
}

// ---- half-GLU gate -----------------------------------------------------------------------
namespace {

struct GluPlan {
    bool tc;
    int splits;
    size_t hdr, Wt, Wn, x1, z, gz, gx1, part, total;
};

GluPlan plan_glu(const ssm_shape& s) {
    GluPlan p{};
    size_t off = 0;
    const size_t M = (size_t)s.B * s.T, HH = (size_t)s.H * s.H;
    p.tc = s.io_dtype == SSM_BF16 && tc_tn_supported((int)M, s.H, s.H, false) && tc_nt_supported(s.H, s.H);
    p.splits = p.tc ? tc_nt_splits((int)M, s.H, s.H) : gemm_nt_splits((int)M, s.H, s.H);
    p.hdr = take(off, sizeof(WsHeader));
    p.Wt = take(off, HH * 4);   // W^T: bf16 planes hi | lo [H, 2H], or fp32
    p.Wn = take(off, p.tc ? 2 * HH * 2 : 0);
    p.x1 = take(off, M * s.H * 4);                  // GELU(v): fp32, or two bf16 planes
    p.z = take(off, M * s.H * 4);                   // the gate's argument
    p.gz = take(off, M * s.H * 4);                  // fp32, or two bf16 planes
    p.gx1 = take(off, M * s.H * 4);
    p.part = take(off, (size_t)2 * p.splits * HH * 4);
    p.total = off;
    return p;
}

}  // namespace

SSM_API size_t ssm_glu_workspace_bytes(const ssm_shape* shape) {
    if (check_shape(shape) != SSM_OK) return 0;
    return plan_glu(*shape).total;
}

SSM_API int ssm_glu_fwd(const ssm_shape* shape, const float* W, const void* v, void* out, void* ws, size_t ws_bytes,
                        void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!W || !v || !out) return SSM_ERR_NULL;
    if (misaligned(W) || misaligned(v) || misaligned(out)) return SSM_ERR_ALIGN;
    const ssm_shape& s = *shape;
    const GluPlan p = plan_glu(s);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const bool bf16 = s.io_dtype == SSM_BF16;
    const int M = s.B * s.T;
    const size_t n = (size_t)M * s.H;
    WsHeader* hdr = at<WsHeader>(ws, p.hdr);
    {
        StageTimer tm("glu_pack_gelu", st);
        launch_glu_pre(bf16, p.tc, n, s.H, v, at<void>(ws, p.x1), W, p.tc ? at<void>(ws, p.Wt) : nullptr, p.tc ? at<void>(ws, p.Wn) : nullptr,
                       p.tc ? nullptr : at<float>(ws, p.Wt), hdr, st);
    }
    {   // z[m, j] = sum_i x1[m, i] W[i, j]
        StageTimer tm("glu_gemm_z", st);
        if (p.tc) {
            // three products of the planes of x1 and W (lo hi, hi lo, hi hi; a single bf16 rounding of x1 here costs
            // 2e-2 on dW); out = v * sigmoid(z) leaves from the same epilogue
            GemmTcTN g{at<void>(ws, p.x1), at<void>(ws, p.Wt), M, s.H, s.H, false, true, at<void>(ws, p.z), nullptr, v, hdr};
            g.gate_out = out;
            g.n_products = 3, g.planes_a = 2, g.planes_w = 2, g.prod_a = 0x001u, g.prod_w = 0x010u;
            if (int rc = launch_gemm_tc_tn(g, st)) return rc;
        } else {
            GemmTN g{at<void>(ws, p.x1), false, s.H, at<void>(ws, p.Wt), false, s.H, M, s.H, s.H, Epi::StoreF32,
                     at<void>(ws, p.z), false, nullptr, nullptr, false, nullptr};
            launch_gemm_tn(g, st);
        }
    }
    if (!p.tc) {
        StageTimer tm("glu_out", st);
        launch_glu_out(bf16, n, v, at<float>(ws, p.z), out, st);
    }
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_glu_bwd(const ssm_shape* shape, const float* W, const void* v, const void* gout, void* ws,
                        size_t ws_bytes, void* gv, float* dW, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!W || !v || !gout || !gv || !dW) return SSM_ERR_NULL;
    if (misaligned(W) || misaligned(v) || misaligned(gout) || misaligned(gv) || misaligned(dW)) return SSM_ERR_ALIGN;
    const ssm_shape& s = *shape;
    const GluPlan p = plan_glu(s);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const bool bf16 = s.io_dtype == SSM_BF16;
    const int M = s.B * s.T;
    const size_t n = (size_t)M * s.H, HH = (size_t)s.H * s.H;
    WsHeader* hdr = at<WsHeader>(ws, p.hdr);
    {
        StageTimer tm("glu_gz", st);
        launch_glu_gz(bf16, p.tc, n, v, gout, at<float>(ws, p.z), at<void>(ws, p.gz), st);
    }
    {   // g_x1[m, i] = sum_j gz[m, j] W[i, j]
        StageTimer tm("glu_gemm_gx1", st);
        if (p.tc) {
            GemmTcTN g{at<void>(ws, p.gz), at<void>(ws, p.Wn), M, s.H, s.H, false, true, at<void>(ws, p.gx1), nullptr, nullptr, hdr};
            g.n_products = 2, g.planes_a = 1, g.planes_w = 2, g.prod_a = 0x00u, g.prod_w = 0x01u;   // gz_hi with lo, then hi
            if (int rc = launch_gemm_tc_tn(g, st)) return rc;
        } else {
            GemmTN g{at<void>(ws, p.gz), false, s.H, W, false, s.H, M, s.H, s.H, Epi::StoreF32,
                     at<void>(ws, p.gx1), false, nullptr, nullptr, false, nullptr};
            launch_gemm_tn(g, st);
        }
    }
    int slices = p.splits;
    {   // dW[i, j] = sum_m x1[m, i] gz[m, j]
        StageTimer tm("glu_gemm_dW", st);
        if (p.tc) {
            // (x1_hi + x1_lo)^T (gz_hi + gz_lo) as two products, one per plane of x1 (column blocks of x1)
            GemmTcNT g0{at<void>(ws, p.x1), 2 * s.H, at<void>(ws, p.gz), at<void>(ws, p.gz + n * 2), at<float>(ws, p.part)};
            GemmTcNT g1 = g0;
            g1.A = at<void>(ws, p.x1 + (size_t)s.H * 2);
            g1.part = at<float>(ws, p.part) + (size_t)p.splits * HH;
            if (int rc = launch_gemm_tc_nt2(M, s.H, s.H, p.splits, g0, g1, hdr, st)) return rc;
            slices *= 2;
        } else {
            const GemmNT g{at<void>(ws, p.x1), false, s.H, at<float>(ws, p.gz), s.H, M, p.splits, at<float>(ws, p.part)};
            launch_gemm_nt(&g, 1, nullptr, st);
        }
    }
    {
        StageTimer tm("glu_gv", st);   // and the sum of dW's slices
        launch_glu_post(bf16, at<float>(ws, p.part), slices, HH, dW, n, v, gout, at<float>(ws, p.z), at<float>(ws, p.gx1), gv, st);
    }
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

// dD's partial sums (rows of [H]) brought down to what the last kernel of the pass adds.
static const float* reduce_dD(const ssm_shape& s, float* part, int* rows, cudaStream_t st) {
    return launch_reduce_rows(part, *rows, s.H, part + (size_t)*rows * s.H, kMaxPartialRows, rows, st);
}

// What a layer's backward pass leaves for its last kernels, which a stack runs for all its layers together.
struct LayerTail {
    GradTail tail;
    GemmTcNtPlanes products[2];   // plane path: the weight-gradient products, not launched yet
    int gA_rows;
};

// Launch sequence of one layer's backward pass, all but its last kernels (layer_bwd_tail).  du_add (fp32 [B,T,H], may
// be NULL) is added to du before it is stored (the gradient of the residual branch of a stacked model).
static int layer_bwd_impl(const ssm_shape& s, const LayerPlan& p, const LayerIo& io, const ssm_c64* Lambda,
                          const float* Delta, const ssm_c64* Bc, const float* D, const void* u, const uint8_t* done,
                          const ssm_c64* x0, const void* gy, const ssm_c64* gxT, const float* du_add, void* ws,
                          WsHeader* hdr, void* du, ssm_c64* dLambda, float* dDelta, ssm_c64* dB, ssm_c64* dC, float* dD,
                          ssm_c64* dx0, LayerTail* left, cudaStream_t st) {
    const int BT = s.B * s.T, P2 = 2 * s.P;
    if (p.tc && !(io.u_bf16 && io.gy_bf16 && io.du_bf16)) return SSM_ERR_DTYPE;
    float* part = at<float>(ws, p.part);                       // split-K partials of gBbar ...
    float* part_c = part + (size_t)p.splits * 2 * s.P * s.H;   // ... and of dC
    const size_t plane = (size_t)BT * s.P * 4;   // bytes of one bf16 plane of a state tensor
    int rc = SSM_OK;
    // The last sums (gAbar over the sequences, dD over row groups, the two split-K sums) are left to the two
    // kernels at the end of the pass: what the stages leave are rows of partial sums.
    const float2* gA_part = nullptr;
    const float* dD_part = nullptr;
    int gA_rows = 0, dD_rows = 0;

    if (p.tc) {
        if (tc_gemm_scan_bwd_supported(s.B, s.T, s.H, s.P)) {
            // projection and reverse scan in one kernel: s = reverse scan(gy conj(C)), g_x stays on chip
            StageTimer tm("gemm_gx_scan_bwd", st);
            GemmScanBwd g{gy, at<void>(ws, p.W1), s.B, s.T, s.H, s.P, at<float2>(ws, p.Abar), at<float>(ws, p.Apow), done, (const float2*)x0,
                          (const float2*)gxT, at<void>(ws, p.xs), at<void>(ws, p.gs), nullptr, (float2*)dx0, hdr};
            if ((rc = launch_gemm_scan_bwd_part(g, at<char>(ws, p.scan), &gA_part, &gA_rows, st))) return rc;
        } else {
            {   // gx[m, 2p+c] = sum_h gy[m,h] conj(C)_c[h,p]   (weights as hi + lo bf16)
                StageTimer tm("gemm_gx", st);
                GemmTcTN g{gy, at<void>(ws, p.W1), BT, P2, s.H, true, true, at<void>(ws, p.f32buf), nullptr, nullptr, hdr};
                if ((rc = launch_gemm_tc_tn(g, st))) return rc;
            }
            {
                StageTimer tm("scan_bwd", st);
                rc = launch_scan_bwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), done,
                                     (const float2*)x0, at<void>(ws, p.xs), true, at<float2>(ws, p.f32buf),
                                     (const float2*)gxT, at<void>(ws, p.gs), true, at<float2>(ws, p.gAbar), (float2*)dx0,
                                     hdr, at<char>(ws, p.scan), st, &gA_part, &gA_rows);
                if (rc) return rc;
            }
        }
        {   // du[m,h] = sum_k s[m,k] Bq[h,k] + D[h] gy[m,h];  where the kernel can, also dD[h] = sum_m gy[m,h] u[m,h]
            // from the tiles of gy its epilogue holds anyway (one more operand tile, u, beside each)
            StageTimer tm("gemm_du", st);
            if (du_add) return SSM_ERR_SHAPE;   // the residual addend exists only on the CUDA-core path (stacks)
            GemmTcTN g{at<void>(ws, p.gs), at<void>(ws, p.W3), BT, s.H, P2, false, false, du, D, gy, hdr};
            if (tc_tn_dot_supported(BT, s.H)) g.dot = u, g.dot_part = at<float>(ws, p.dot), g.dot_rows = &dD_rows;
            if ((rc = launch_gemm_tc_tn(g, st))) return rc;
            if (g.dot) dD_part = reduce_dD(s, g.dot_part, &dD_rows, st);
        }
        {   // gBbar[p,h] = sum_m s[m,p] u[m,h] and dC[h,p] = sum_m gy[m,h] conj(x[m,p])
            StageTimer tm("gemm_gBbar_gC", st);
            const GemmTcNT gB{u, s.H, at<void>(ws, p.gs), at<void>(ws, p.gs + plane), part};
            const GemmTcNT gC{gy, s.H, at<void>(ws, p.xs), at<void>(ws, p.xs + plane), part_c};
            if ((rc = launch_gemm_tc_nt2(BT, s.H, P2, p.splits, gB, gC, hdr, st))) return rc;
        }
    } else if (p.planes) {
        const bool gyb = io.gy_bf16, ub = io.u_bf16;
        if (!gyb && tc_tile_scan_supported(s.B, s.T, s.H, s.P, false)) {
            StageTimer tm("scan_bwd", st);   // g_x as below, scanned in the projection's epilogue
            TileScan scan{s.B, s.T, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), done, (const float2*)x0, (const float2*)gxT, nullptr, (float2*)dx0,
                          at<float2>(ws, p.xs)};
            GemmTcTN g{gy, at<void>(ws, p.W1), BT, P2, s.H, false, true, at<void>(ws, p.gs), nullptr, nullptr, hdr};
            g.scan = &scan;
            scan.gA_part = scan_partials(at<char>(ws, p.scan));
            if ((rc = plane_projection(g, false, at<void>(ws, p.gy3), true, st))) return rc;
            gA_part = reduce_scan_partials(s.B, s.P, at<char>(ws, p.scan), &gA_rows, st);
        } else {
        {   // g_x = gy conj(C)
            StageTimer tm("gemm_gx", st);
            const GemmTcTN g{gy, at<void>(ws, p.W1), BT, P2, s.H, false, true, at<void>(ws, p.gs), nullptr, nullptr, hdr};
            if ((rc = plane_projection(g, gyb, at<void>(ws, p.gy3), true, st))) return rc;
        }
        {
            StageTimer tm("scan_bwd", st);
            rc = launch_scan_bwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), done, (const float2*)x0,
                                 at<void>(ws, p.xs), false, at<float2>(ws, p.gs), (const float2*)gxT,
                                 at<void>(ws, p.gs), false, at<float2>(ws, p.gAbar), (float2*)dx0, hdr,
                                 at<char>(ws, p.scan), st, &gA_part, &gA_rows);
            if (rc) return rc;
        }
        }
        {   // du = s Bq^T + D gy (+ the residual branch's gradient), and dD's sums
            StageTimer tm("gemm_du", st);
            GemmTcTN g{at<void>(ws, p.gs), at<void>(ws, p.W3), BT, s.H, P2, false, !io.du_bf16, du, D, gy, hdr};
            g.skip_bf16 = gyb, g.add = du_add;
            g.dot = u, g.dot_bf16 = ub, g.dot_part = at<float>(ws, p.dot), g.dot_rows = &dD_rows;
            if ((rc = plane_projection(g, false, at<void>(ws, p.s3), true, st))) return rc;
            dD_part = reduce_dD(s, g.dot_part, &dD_rows, st);
        }
        // gBbar = s^T u and dC = gy^T conj(x)
        left->products[0] = {ub ? u : at<void>(ws, p.u3), at<void>(ws, p.s3), ub ? 1 : 3, 3, ub ? 3 : 6, ub ? kProd3A : kProd6A,
                             ub ? kProd3B : kProd6B, part};
        left->products[1] = {gyb ? gy : at<void>(ws, p.gy3), at<void>(ws, p.x3), gyb ? 1 : 3, 3, gyb ? 3 : 6,
                             gyb ? kProd3A : kProd6A, gyb ? kProd3B : kProd6B, part_c};
    } else {
        {
            StageTimer tm("gemm_gx", st);
            GemmTN g3{gy, io.gy_bf16, s.H, at<void>(ws, p.W1), false, s.H, BT, P2, s.H, Epi::StoreF32,
                      at<void>(ws, p.gs), false, nullptr, nullptr, false, nullptr};
            launch_gemm_tn(g3, st);
        }
        {
            StageTimer tm("scan_bwd", st);
            rc = launch_scan_bwd(s.B, s.T, s.P, at<float2>(ws, p.Abar), at<float2>(ws, p.Alo), done, (const float2*)x0,
                                 at<void>(ws, p.xs), false, at<float2>(ws, p.gs), (const float2*)gxT,
                                 at<void>(ws, p.gs), false, at<float2>(ws, p.gAbar), (float2*)dx0, hdr,
                                 at<char>(ws, p.scan), st, &gA_part, &gA_rows);
            if (rc) return rc;
        }
        {
            StageTimer tm("gemm_du", st);
            GemmTN g4{at<void>(ws, p.gs), false, P2, at<void>(ws, p.W3), false, P2, BT, s.H, P2, Epi::AddDiagIo,
                      du, io.du_bf16, D, gy, io.gy_bf16, du_add};
            launch_gemm_tn(g4, st);
        }
        {   // both weight gradients, and the row groups' sums of gy * u for dD
            StageTimer tm("gemm_gBbar_gC", st);
            const GemmNT g[2] = {{u, io.u_bf16, s.H, at<float>(ws, p.gs), P2, BT, p.splits, part},
                                 {gy, io.gy_bf16, s.H, at<float>(ws, p.xs), P2, BT, p.splits, part_c}};
            const SimtDot dot{gy, u, io.gy_bf16, io.u_bf16, at<float>(ws, p.dot)};
            launch_gemm_nt(g, 2, &dot, st);
            dD_rows = dot_groups(BT);
            dD_part = reduce_dD(s, at<float>(ws, p.dot), &dD_rows, st);
        }
    }
    if (!dD_part) {   // dD[h] = sum_m gy[m,h] u[m,h], unless the du projection left its partial sums already
        StageTimer tm("dot_gy_u", st);
        float* tmp = at<float>(ws, p.dot);
        int groups = launch_dot_columns_partial(io.gy_bf16, gy, io.u_bf16, u, BT, s.H, tmp, st);
        dD_part = launch_reduce_rows(tmp, groups, s.H, tmp + (size_t)groups * s.H, kMaxPartialRows, &dD_rows, st);
    }
    left->gA_rows = gA_rows;
    left->tail = {(const float2*)Lambda, Delta, (const float2*)Bc, part, part_c, (float2*)dB, (float2*)dC, at<float2>(ws, p.gg),
                  gA_part, (float2*)dLambda, dDelta, {dD_part, nullptr, nullptr}, {dD_rows, 0, 0}, {dD, nullptr, nullptr}};
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

// The weight-gradient products of the plane path, the sums over split-K partials and the adjoint of the discretisation
// (with the sums of gAbar, dD and a stack's LayerNorm parameters) of n layers of one shape.
static int layer_bwd_tail(const ssm_shape& s, const LayerPlan& p, int n, const LayerTail* left, WsHeader* hdr, cudaStream_t st) {
    GemmTcNtPlanes products[2 * kMaxStackLayers];
    GradTail tails[kMaxStackLayers];
    for (int l = 0; l < n; ++l) {
        products[2 * l] = left[l].products[0];
        products[2 * l + 1] = left[l].products[1];
        tails[l] = left[l].tail;
    }
    int splits = p.splits;
    if (p.planes) {
        StageTimer tm("gemm_gBbar_gC", st);
        splits = std::min(splits, tc_nt_planes_splits(s.B * s.T, s.H, 2 * s.P, 2 * n));
        if (int rc = launch_gemm_tc_nt_planes(s.B * s.T, s.H, 2 * s.P, splits, 2 * n, products, hdr, st)) return rc;
    }
    StageTimer tm("gD_and_discretize_bwd", st);
    launch_layer_tail(s.H, s.P, splits, n, tails, left[0].gA_rows, st);
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_layer_bwd(const ssm_shape* shape, const ssm_c64* Lambda, const float* Delta, const ssm_c64* Bc,
                          const ssm_c64* Cc, const float* D, const void* u, const uint8_t* done,
                          const ssm_c64* x0, const void* gy, const ssm_c64* gxT, void* ws, size_t ws_bytes,
                          void* du, ssm_c64* dLambda, float* dDelta, ssm_c64* dB, ssm_c64* dC, float* dD,
                          ssm_c64* dx0, void* stream) {
    if (int rc = check_shape(shape)) return rc;
    if (!Lambda || !Delta || !Bc || !Cc || !D || !u || !gy || !du || !dLambda || !dDelta || !dB || !dC || !dD)
        return SSM_ERR_NULL;
    if (misaligned(Lambda) || misaligned(Delta) || misaligned(Bc) || misaligned(Cc) || misaligned(D) ||
        misaligned(u) || misaligned(gy) || misaligned(du) || misaligned(dLambda) || misaligned(dDelta) ||
        misaligned(dB) || misaligned(dC) || misaligned(dD) || misaligned(x0) || misaligned(gxT) || misaligned(dx0))
        return SSM_ERR_ALIGN;
    const ssm_shape& s = *shape;
    const LayerPlan p = plan_layer(s);
    if (int rc = check_ws(ws, ws_bytes, p.total)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    WsHeader* hdr = at<WsHeader>(ws, p.hdr);
    LayerTail left{};
    if (p.small) {
        {
            StageTimer tm("scan_bwd", st);   // (with everything around the scan)
            float* part = at<float>(ws, p.part);
            left.gA_rows = s.B;
            left.tail = {(const float2*)Lambda, Delta, (const float2*)Bc, part, part + (size_t)p.splits * 2 * s.P * s.H, (float2*)dB,
                         (float2*)dC, at<float2>(ws, p.gg), at<float2>(ws, p.scan), (float2*)dLambda, dDelta,
                         {at<float>(ws, p.dot), nullptr, nullptr}, {s.B, 0, 0}, {dD, nullptr, nullptr}};
            const LayerSmall g{s.B, s.T, s.H, s.P, s.io_dtype == SSM_BF16, (const float2*)Lambda, Delta, (const float2*)Bc,
                               (const float2*)Cc, D, u, done, (const float2*)x0, (const float2*)gxT, gy, at<float2>(ws, p.xs), du, nullptr,
                               (float2*)dx0, hdr};
            if (int rc = launch_layer_small_bwd(g, left.tail, p.slices ? nullptr : at<float2>(ws, p.gs), at<float2>(ws, p.scan), at<float>(ws, p.dot), st))
                return rc;
        }
        if (!p.slices) {
            StageTimer tm("gemm_gBbar_gC", st);
            const int BT = s.B * s.T, P2 = 2 * s.P;
            const bool b = s.io_dtype == SSM_BF16;
            const GemmNT g[2] = {{u, b, s.H, at<float>(ws, p.gs), P2, BT, p.splits, const_cast<float*>(left.tail.part_b)},
                                 {gy, b, s.H, at<float>(ws, p.xs), P2, BT, p.splits, const_cast<float*>(left.tail.part_c)}};
            launch_gemm_nt(g, 2, nullptr, st, true);
        }
        if (s.B > 1) return layer_bwd_tail(s, p, 1, &left, hdr, st);
        SSM_RETURN_IF_CUDA_ERROR();
        return SSM_OK;
    }
    if (int rc = layer_bwd_impl(s, p, layer_io(s), Lambda, Delta, Bc, D, u, done, x0, gy, gxT, nullptr, ws, hdr, du, dLambda,
                                dDelta, dB, dC, dD, dx0, &left, st))
        return rc;
    return layer_bwd_tail(s, p, 1, &left, hdr, st);
}

// ---- stacked model -----------------------------------------------------------------------------
namespace {

// Storage inside a stack.  Only the stack's input u, its output, gout and du are in the I/O type.
// Everything that passes between the layers (the SSM outputs v, the layer inputs, the gradients
// handed from a layer to the one below) is fp32: stored in bf16, a value that rounds to the other
// neighbour than in an exact evaluation is a legitimate difference between two correct runs, and the
// layers that follow amplify such differences in the parameter-gradient sums beyond the tolerance of
// the I/O type.  The layers therefore run with fp32 inputs and outputs (except for the first layer's
// input and the last gradient), on the fp32 path of the layer.
struct StackPlan {
    size_t layer_ws;   // bytes of one layer workspace
    size_t act;        // bytes of one fp32 [B,T,H] tensor
    size_t hdr, layers, acts, vs, stats, gz, gv, g0, g1, tmp, tmp_stride, total;
};

ssm_shape stack_layer_shape(const ssm_shape& s) {
    ssm_shape t = s;
    t.io_dtype = SSM_F32;
    return t;
}

StackPlan plan_stack(const ssm_shape& s, int L) {
    StackPlan p{};
    size_t off = 0;
    const size_t BT = (size_t)s.B * s.T;
    p.layer_ws = align_up(plan_layer(stack_layer_shape(s), false).total, 256);
    p.act = align_up(BT * s.H * 4, 256);
    p.hdr = take(off, sizeof(WsHeader));
    p.layers = take(off, p.layer_ws * L);
    p.acts = take(off, p.act * (L > 1 ? L - 1 : 0));   // inputs of layers 1 .. L-1
    p.vs = take(off, p.act * L);                       // SSM outputs
    p.stats = take(off, align_up(BT * 4, 256) * 2 * L);   // mean and 1/std of every row, per layer
    p.gz = take(off, p.act);
    p.gv = take(off, p.act);
    p.g0 = take(off, p.act);
    p.g1 = take(off, p.act);
    p.tmp_stride = align_up(stack_tmp_floats((int)BT, s.H) * 4, 256);
    p.tmp = take(off, p.tmp_stride * L);
    p.total = off;
    return p;
}

int check_stack_args(const ssm_shape* shape, int n_layers, const ssm_stack_params* params) {
    if (int rc = check_shape(shape)) return rc;
    if (n_layers < 1 || n_layers > kMaxStackLayers) return SSM_ERR_SHAPE;
    if (!params) return SSM_ERR_NULL;
    for (int l = 0; l < n_layers; ++l) {
        const ssm_stack_params& q = params[l];
        if (!q.Lambda || !q.Delta || !q.Bc || !q.Cc || !q.D || !q.ln_weight || !q.ln_bias) return SSM_ERR_NULL;
        if (misaligned(q.Lambda) || misaligned(q.Delta) || misaligned(q.Bc) || misaligned(q.Cc) || misaligned(q.D) ||
            misaligned(q.ln_weight) || misaligned(q.ln_bias))
            return SSM_ERR_ALIGN;
    }
    return SSM_OK;
}

}  // namespace

SSM_API size_t ssm_stack_workspace_bytes(const ssm_shape* shape, int n_layers) {
    if (check_shape(shape) != SSM_OK || n_layers < 1 || n_layers > kMaxStackLayers) return 0;
    return plan_stack(*shape, n_layers).total;
}

SSM_API int ssm_stack_fwd(const ssm_shape* shape, int n_layers, const ssm_stack_params* params, const void* u,
                          const uint8_t* done, void* out, void* ws, size_t ws_bytes, void* stream) {
    if (int rc = check_stack_args(shape, n_layers, params)) return rc;
    if (!u || !out) return SSM_ERR_NULL;
    if (misaligned(u) || misaligned(out)) return SSM_ERR_ALIGN;
    const ssm_shape& s = *shape;
    const StackPlan sp = plan_stack(s, n_layers);
    if (int rc = check_ws(ws, ws_bytes, sp.total)) return rc;
    const ssm_shape ls = stack_layer_shape(s);
    const LayerPlan lp = plan_layer(ls, false);
    cudaStream_t st = (cudaStream_t)stream;
    const bool bf16 = s.io_dtype == SSM_BF16;
    const int BT = s.B * s.T;
    const size_t stat = align_up((size_t)BT * 4, 256);
    WsHeader* hdr = at<WsHeader>(ws, sp.hdr);
    {   // the parameters of all layers in one launch
        StageTimer tm("discretize_pack", st);
        PackJob jobs[kMaxStackLayers];
        for (int l = 0; l < n_layers; ++l)
            jobs[l] = pack_job(lp, params[l].Lambda, params[l].Delta, params[l].Bc, params[l].Cc, at<void>(ws, sp.layers + sp.layer_ws * l));
        if (lp.planes) launch_discretize_pack_planes(ls.H, ls.P, n_layers, jobs, hdr, st);
        else launch_discretize_pack_f32(ls.H, ls.P, n_layers, jobs, hdr, st);
    }
    const void* in = u;
    for (int l = 0; l < n_layers; ++l) {
        const ssm_stack_params& q = params[l];
        const bool first = l == 0, last = l == n_layers - 1;
        void* lws = at<void>(ws, sp.layers + sp.layer_ws * l);
        float* v = at<float>(ws, sp.vs + sp.act * l);
        void* o = last ? out : at<void>(ws, sp.acts + sp.act * l);
        const LayerIo io{first && bf16, false, false, false};
        if (int rc = layer_fwd_run(ls, lp, io, q.D, in, done, nullptr, v, nullptr, lws, hdr, true, st))
            return rc;
        StageTimer tm("stack_gelu_ln_fwd", st);
        launch_stack_fwd(first && bf16, last && bf16, BT, s.H, in, v, q.ln_weight, q.ln_bias, o,
                         at<float>(ws, sp.stats + stat * (2 * l)), at<float>(ws, sp.stats + stat * (2 * l + 1)), st);
        in = o;
    }
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}

SSM_API int ssm_stack_bwd(const ssm_shape* shape, int n_layers, const ssm_stack_params* params, const void* u,
                          const uint8_t* done, const void* gout, void* ws, size_t ws_bytes, void* du,
                          const ssm_stack_grads* grads, void* stream) {
    if (int rc = check_stack_args(shape, n_layers, params)) return rc;
    if (!u || !gout || !du || !grads) return SSM_ERR_NULL;
    if (misaligned(u) || misaligned(gout) || misaligned(du)) return SSM_ERR_ALIGN;
    for (int l = 0; l < n_layers; ++l) {
        const ssm_stack_grads& g = grads[l];
        if (!g.dLambda || !g.dDelta || !g.dB || !g.dC || !g.dD || !g.dln_weight || !g.dln_bias) return SSM_ERR_NULL;
        if (misaligned(g.dLambda) || misaligned(g.dDelta) || misaligned(g.dB) || misaligned(g.dC) || misaligned(g.dD) ||
            misaligned(g.dln_weight) || misaligned(g.dln_bias))
            return SSM_ERR_ALIGN;
    }
    const ssm_shape& s = *shape;
    const StackPlan sp = plan_stack(s, n_layers);
    if (int rc = check_ws(ws, ws_bytes, sp.total)) return rc;
    const ssm_shape ls = stack_layer_shape(s);
    const LayerPlan lp = plan_layer(ls, false);
    cudaStream_t st = (cudaStream_t)stream;
    const bool bf16 = s.io_dtype == SSM_BF16;
    const int BT = s.B * s.T;
    const size_t stat = align_up((size_t)BT * 4, 256);
    WsHeader* hdr = at<WsHeader>(ws, sp.hdr);
    const void* g = gout;
    LayerTail left[kMaxStackLayers] = {};
    for (int l = n_layers - 1; l >= 0; --l) {
        const ssm_stack_params& q = params[l];
        const ssm_stack_grads& gr = grads[l];
        const bool first = l == 0, top = l == n_layers - 1;
        void* lws = at<void>(ws, sp.layers + sp.layer_ws * l);
        const void* in = first ? u : at<void>(ws, sp.acts + sp.act * (l - 1));
        const float* v = at<float>(ws, sp.vs + sp.act * l);
        void* gnext = first ? du : at<void>(ws, (l & 1) ? sp.g1 : sp.g0);
        const float *dw_part = nullptr, *db_part = nullptr;
        int ln_rows = 0;
        {
            StageTimer tm("stack_gelu_ln_bwd", st);
            launch_stack_bwd(top && bf16, first && bf16, BT, s.H, g, in, v, q.ln_weight,
                             at<float>(ws, sp.stats + stat * (2 * l)), at<float>(ws, sp.stats + stat * (2 * l + 1)),
                             at<float>(ws, sp.gz), at<float>(ws, sp.gv), at<float>(ws, sp.tmp + sp.tmp_stride * l), &dw_part,
                             &db_part, &ln_rows, st);
        }
        // the gradient handed down: gz (residual branch) + du of the SSM, summed in fp32 in the du epilogue
        const LayerIo io{first && bf16, false, false, first && bf16};
        if (int rc = layer_bwd_impl(ls, lp, io, q.Lambda, q.Delta, q.Bc, q.D, in, done, nullptr, at<void>(ws, sp.gv), nullptr,
                                    at<float>(ws, sp.gz), lws, hdr, gnext, gr.dLambda, gr.dDelta, gr.dB, gr.dC, gr.dD,
                                    nullptr, &left[l], st))
            return rc;
        GradTail& t = left[l].tail;
        t.sum_part[1] = dw_part, t.sum_part[2] = db_part;
        t.sum_rows[1] = t.sum_rows[2] = ln_rows;
        t.sum_out[1] = gr.dln_weight, t.sum_out[2] = gr.dln_bias;
        g = gnext;
    }
    // What no other layer waits for, for all layers together.
    if (int rc = layer_bwd_tail(ls, lp, n_layers, left, hdr, st)) return rc;
    SSM_RETURN_IF_CUDA_ERROR();
    return SSM_OK;
}
