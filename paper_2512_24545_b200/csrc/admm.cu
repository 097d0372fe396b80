// ADMM refinement of one MDBF factor with the other held fixed (Section "ADMM Refinement"):
//
//     U_tilde = (W V + rho (U - Lam)) (V^T V + rho I)^-1        Eq. admm-U-tilde
//     U       = MSVID_l[U_tilde + Lam]                          Eq. admm-U-prox
//     Lam     = Lam + U_tilde - U                               Eq. admm-U-dual
//
// W is N x M, V is M x R, U and Lam are N x R (dense values of the factor), all fp32 row-major on the device.  The
// update of the other factor is the same call on the transposed problem (transpose_w).
//
// The two dense products (W V and V^T V, once per call) run on the tensor cores at close to fp32 accuracy (gemm3x.cu: scaled
// fp16 operands in a three-term split); V's operand images serve both, as the right operand of W V and as both operands of
// V^T V.  The Cholesky factorisation of the R x R system (cuSOLVER) is the one library routine; its factor is inverted here by
// doubling, the inverse of the system is formed and then applied, in every inner iteration, by the same tensor-core product.
// Everything specific to the method is this library's own: the MSVID step (mdbf_msvid: sign mask + rank-l envelope on the tensor
// cores), the elementwise passes around it, and the reconstruction of the dense factor from the compact one fused with
// the dual update.
//
// The system is symmetric, so the column-major solver works on the row-major memory as it is; what it calls the lower
// triangle are the rows above the diagonal here.
#include <cusolverDn.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"

namespace mdbf {
namespace admm {

struct Libs {
    cusolverDnHandle_t solver = nullptr;
    float *potrf_ws = nullptr;          // the factorisation's scratch, as large as the largest request so far
    int potrf_floats = 0;
    int device = -1;
    cudaStream_t side = nullptr;        // the R x R system is factored and inverted here while W V runs on the caller's stream
    cudaEvent_t fork = nullptr, join = nullptr;
};
static thread_local Libs g_libs;

static mdbf_status_t get_libs(int device, cudaStream_t st, Libs **out) {
    Libs &L = g_libs;
    if (L.device != device) {
        if (L.solver) cusolverDnDestroy(L.solver);
        if (L.potrf_ws) cudaFree(L.potrf_ws);
        if (L.side) cudaStreamDestroy(L.side);
        if (L.fork) cudaEventDestroy(L.fork);
        if (L.join) cudaEventDestroy(L.join);
        L = Libs();
        if (cusolverDnCreate(&L.solver) != CUSOLVER_STATUS_SUCCESS) {
            L = Libs();
            set_error("cusolverDnCreate failed");
            return MDBF_ERR_CUDA;
        }
        if (cudaStreamCreateWithFlags(&L.side, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&L.fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&L.join, cudaEventDisableTiming) != cudaSuccess ||
            cusolverDnSetStream(L.solver, L.side) != CUSOLVER_STATUS_SUCCESS) {
            cusolverDnDestroy(L.solver);
            if (L.side) cudaStreamDestroy(L.side);
            if (L.fork) cudaEventDestroy(L.fork);
            if (L.join) cudaEventDestroy(L.join);
            L = Libs();
            set_error("could not create the side stream of the refinement step");
            return MDBF_ERR_CUDA;
        }
        L.device = device;
    }
    (void)st;
    *out = &L;
    return MDBF_OK;
}

// the solver's scratch, as large as the largest request so far
static mdbf_status_t grow_scratch(Libs *L, int floats, cudaStream_t st, const char *who) {
    if (floats <= L->potrf_floats) return MDBF_OK;
    MDBF_CUDA(cudaStreamSynchronize(st));                         // the stream that uses it: the old scratch may still be in use
    if (L->potrf_ws) cudaFree(L->potrf_ws);
    L->potrf_ws = nullptr;
    L->potrf_floats = 0;
    if (dev_malloc(&L->potrf_ws, (size_t)floats * sizeof(float)) != cudaSuccess) {
        set_error("%s: out of device memory for the solver's scratch (%zu bytes)", who, (size_t)floats * sizeof(float));
        return MDBF_ERR_CUDA;
    }
    L->potrf_floats = floats;
    return MDBF_OK;
}

__global__ void ridge_kernel(float *__restrict__ G, int r, float rho) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < r) G[(size_t)i * r + i] += rho;
}

// ------------------------------------------------------------------ Y = U^-1, U upper triangular (r x r, row-major)
// By doubling: the diagonal blocks of TI_LEAF columns are inverted all at once, then neighbouring inverses Y11, Y22 are joined,
//     [U11 U12]^-1   [Y11  -Y11 U12 Y22]
//     [     U22]   = [          Y22    ],
// all pairs of a size in two batched products: log2(r / TI_LEAF) levels instead of the r / 256 dependent steps of a triangular solve
// with r right-hand sides (r = 3712: 2.6 ms of such steps in the library's solver, 0.5 ms here).  Pairs of blocks of
// TI_DENSE columns and more go through the tensor-core product.
constexpr int TI_LEAF = 64, TI_DENSE = 1024;                     // leaves of 128: 45 us longer at r = 3712, of 32: the same
constexpr int TI_SMEM = 2 * TI_LEAF * (TI_LEAF + 1) * 4;
// CTA = one diagonal block, thread = column of the inverse, back substitution: the row of U is the same for the whole warp (a
// broadcast), the column of Y is the thread's own.  The block's lower triangle is written as zeros.
__global__ void __launch_bounds__(TI_LEAF) tri_leaf_kernel(const float *__restrict__ U, float *__restrict__ Y, int r) {
    extern __shared__ float ti_smem[];
    float (*us)[TI_LEAF + 1] = reinterpret_cast<float (*)[TI_LEAF + 1]>(ti_smem);
    float (*ys)[TI_LEAF + 1] = us + TI_LEAF;
    const int o = blockIdx.x * TI_LEAF, j = threadIdx.x, s = min(TI_LEAF, r - o);
    for (int i = 0; i < TI_LEAF; ++i) us[i][j] = (i < s && j < s && j >= i) ? U[(size_t)(o + i) * r + o + j] : (i == j ? 1.f : 0.f);
    __syncthreads();
    for (int i = TI_LEAF - 1; i >= 0; --i) {
        float a[4] = {i == j ? 1.f : 0.f, 0.f, 0.f, 0.f};
        int k = i + 1;
        for (; k + 4 <= TI_LEAF; k += 4)
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = fmaf(-us[i][k + u], ys[k + u][j], a[u]);
        for (; k < TI_LEAF; ++k) a[0] = fmaf(-us[i][k], ys[k][j], a[0]);
        ys[i][j] = i <= j ? ((a[0] + a[1]) + (a[2] + a[3])) / us[i][i] : 0.f;
    }
    if (j < s)
        for (int i = 0; i < s; ++i) Y[(size_t)(o + i) * r + o + j] = ys[i][j];
}
// One of the two products that join the pairs of blocks of s columns (blockIdx.z = pair): out = A B (FIRST: A = U12, B = Y22; P) or
// -A B (A = Y11, B = P; Y12), fp32 on the CUDA cores: 64 x 64 tiles, 256 threads of 4 x 4, the triangular operand's zeros skipped.
template <bool FIRST>
__global__ void __launch_bounds__(256) tri_join_kernel(const float *__restrict__ A, const float *__restrict__ B, float *__restrict__ out, int r, int s) {
    __shared__ __align__(16) float as[16][68], bs[16][68];       // [k][row], [k][column]
    const int o = blockIdx.z * 2 * s, s2 = min(s, r - o - s);
    const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64;
    if (j0 >= s2) return;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const float *a = A + (size_t)o * r + (FIRST ? o + s : o);                                // U12 (s x s2) or Y11 (s x s)
    const float *b = FIRST ? B + (size_t)(o + s) * r + o + s : B + (size_t)o * r + o + s;    // Y22 (s2 x s2) or P (s x s2)
    const int depth = FIRST ? s2 : s;
    const int k_lo = FIRST ? 0 : i0, k_hi = FIRST ? min(depth, j0 + 64) : depth;             // Y22[k][j] = 0 for k > j, Y11[i][k] = 0 for k < i
    float acc[4][4] = {};
    for (int k0 = k_lo; k0 < k_hi; k0 += 16) {
        {
            const int kk = tid & 15;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int row = (tid >> 4) + 16 * u;
                as[kk][row] = (i0 + row < s && k0 + kk < k_hi) ? a[(size_t)(i0 + row) * r + k0 + kk] : 0.f;
                const int col = tid & 63, kb = (tid >> 6) + 4 * u;
                bs[kb][col] = (k0 + kb < k_hi && j0 + col < s2) ? b[(size_t)(k0 + kb) * r + j0 + col] : 0.f;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float4 x = *reinterpret_cast<const float4 *>(&as[k][4 * ty]), y = *reinterpret_cast<const float4 *>(&bs[k][4 * tx]);
            const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(xa[p], yb[q], acc[p][q]);
        }
        __syncthreads();
    }
    float *dst = out + (size_t)o * r + o + s;
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i0 + 4 * ty + p < s && j0 + 4 * tx + q < s2) dst[(size_t)(i0 + 4 * ty + p) * r + j0 + 4 * tx + q] = FIRST ? acc[p][q] : -acc[p][q];
}
// U (upper triangle read) -> Y (r x r, written whole); P: r x r scratch, img: operand images of the two blocks of a
// product, s and at most s rows by s at most (s the largest power of two times TI_LEAF below r: 2048 and 1664 at r = 3712), which r x r images hold
static mdbf_status_t tri_inverse(const float *U, float *Y, float *P, uint32_t *img, int r, int32_t *status, cudaStream_t st) {
    static PerDeviceOnce once;
    if (auto first = once.first()) MDBF_CUDA(cudaFuncSetAttribute(tri_leaf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TI_SMEM));
    MDBF_CUDA(cudaMemsetAsync(Y, 0, (size_t)r * r * sizeof(float), st));
    tri_leaf_kernel<<<ceil_div(r, TI_LEAF), TI_LEAF, TI_SMEM, st>>>(U, Y, r);
    for (int s = TI_LEAF; s < r; s *= 2) {
        const int pairs = ceil_div(r - s, 2 * s);                // pairs whose second block is not empty
        if (s < TI_DENSE) {
            const dim3 grid(ceil_div(s, 64), ceil_div(s, 64), pairs);
            tri_join_kernel<true><<<grid, 256, 0, st>>>(U, Y, P, r, s);
            tri_join_kernel<false><<<grid, 256, 0, st>>>(Y, P, Y, r, s);
            continue;
        }
        for (int p = 0; p < pairs; ++p) {
            const int o = p * 2 * s, s2 = std::min(s, r - o - s);
            const size_t d11 = (size_t)o * r + o, d12 = d11 + s, d22 = (size_t)(o + s) * r + o + s;
            uint32_t *a = img, *b = img + gemm3x_image_bytes(s, s) / 4;
            mdbf_status_t rc = gemm3x_split(U + d12, (size_t)r, 1, s, s2, a, st);                      // P = U12 Y22
            if (rc == MDBF_OK) rc = gemm3x_split(Y + d22, 1, (size_t)r, s2, s2, b, st);
            if (rc == MDBF_OK) rc = gemm3x_run(a, b, G3xOut{P + d12, r, false, nullptr, nullptr}, s, s2, s2, status, st);
            if (rc == MDBF_OK) rc = gemm3x_split(Y + d11, (size_t)r, 1, s, s, a, st);                  // Y12 = -Y11 P
            if (rc == MDBF_OK) rc = gemm3x_split(P + d12, 1, (size_t)r, s2, s, b, st);
            if (rc == MDBF_OK) rc = gemm3x_run(a, b, G3xOut{Y + d12, r, true, nullptr, nullptr}, s, s2, s, status, st);
            if (rc) return rc;
        }
    }
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}
// U = S (.) (Ul Vl^T) entry by entry from the compact MSVID result, and Lam += U_tilde - U (Eq. admm-U-dual, rounded as written: near
// convergence U_tilde - U and Lam are small beside Z = U_tilde + Lam, and Z - U would carry a rounding of Z into the dual in every
// iteration; 8192 x 3712 at the end of a refinement, error of the dual step relative to the dual: 1.4e-6 with Z - U, below 6e-8 this way).
// Bound by memory (U_tilde and Lam read, U and Lam written: 16 bytes per entry; 8192 x 3712, l = 16: 130 us, of which the traffic needs
// 74; four rows in flight and 64 registers: 121, but it spills).  CTA = 32 rows x 256 columns; thread = column (its row of Vl in
// registers), the rows' Ul in shared memory, eight rows' loads in flight together; L = l rounded up to 4, 8, 16 or 32.  Ut may be U itself:
// an entry is read by the thread that writes it.
constexpr int RC_ROWS = 32, RC_COLS = 256, RC_BATCH = 8;
template <int L>
__global__ void __launch_bounds__(RC_COLS) recon_dual_kernel(const uint32_t *__restrict__ S, const float *__restrict__ Ul,
                                                             const float *__restrict__ Vl, int l, const float *Ut, float *U,
                                                             float *__restrict__ Lam, int n, int r, int nwords) {
    __shared__ __align__(16) float us[RC_ROWS][L];
    const int i0 = blockIdx.y * RC_ROWS;
    for (int e = threadIdx.x; e < RC_ROWS * L; e += RC_COLS) {
        const int i = e / L, t = e - i * L;
        us[i][t] = (i0 + i < n && t < l) ? Ul[(size_t)(i0 + i) * l + t] : 0.f;
    }
    __syncthreads();
    const int j = blockIdx.x * RC_COLS + threadIdx.x;
    if (j >= r) return;
    float v[L];
#pragma unroll
    for (int t = 0; t < L; ++t) v[t] = t < l ? Vl[(size_t)j * l + t] : 0.f;
    float ut[RC_BATCH], lm[RC_BATCH];
    uint32_t word[RC_BATCH];
    auto load = [&](int ib) {
#pragma unroll
        for (int u = 0; u < RC_BATCH; ++u) {
            const int i = min(i0 + ib + u, n - 1);
            ut[u] = Ut[(size_t)i * r + j];
            lm[u] = Lam[(size_t)i * r + j];
            word[u] = S[(size_t)i * nwords + (j >> 5)];
        }
    };
    load(0);
#pragma unroll 1
    for (int ib = 0; ib < RC_ROWS && i0 + ib < n; ib += RC_BATCH) {
        float val[RC_BATCH], lam[RC_BATCH];
#pragma unroll
        for (int u = 0; u < RC_BATCH; ++u) {
            float e = 0.f;
#pragma unroll
            for (int t = 0; t < L; t += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(&us[ib + u][t]);
                e = fmaf(a.x, v[t], fmaf(a.y, v[t + 1], fmaf(a.z, v[t + 2], fmaf(a.w, v[t + 3], e))));
            }
            val[u] = ((word[u] >> (j & 31)) & 1u) ? -e : e;
            lam[u] = lm[u] + (ut[u] - val[u]);
        }
        if (ib + RC_BATCH < RC_ROWS && i0 + ib + RC_BATCH < n) load(ib + RC_BATCH);      // the next rows' loads run under these stores
#pragma unroll
        for (int u = 0; u < RC_BATCH; ++u)
            if (i0 + ib + u < n) {
                const size_t at = (size_t)(i0 + ib + u) * r + j;
                U[at] = val[u];
                Lam[at] = lam[u];
            }
    }
}
// a failed factorisation (not expected: the system is positive definite for rho > 0) or an expired wait of the product
// kernel turns the singular values into NaN
__global__ void flag_kernel(const int *__restrict__ info, float *__restrict__ sigma, int l) {
    if ((info[0] != 0 || info[2] != 0) && threadIdx.x < l) sigma[threadIdx.x] = __int_as_float(0x7fc00000);
}

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
struct Scratch {
    float *B0, *T, *Z, *G;      // T: scratch of the triangular inverse
    uint32_t *Wimg, *Vimg;      // operand images of op(W) (N row tiles, M deep) and of V^T (R row tiles, M deep)
    uint32_t *Yimg;             // images of L^-T (R x R), formed on the side stream while W's are in use
    int *info;                  // [0], [1]: the solver's; [2]: status word of the product kernel
    char *msvid;
    size_t msvid_bytes;
};
static mdbf_status_t carve(Scratch *w, char *base, int64_t n, int64_t m, int64_t r, int32_t l, size_t *total) {
    size_t msv = 0;
    mdbf_status_t rc = mdbf_msvid_workspace_bytes(n, r, l, &msv);
    if (rc) return rc;
    size_t off = 0;
    auto take = [&](size_t bytes) { char *p = base ? base + off : nullptr; off += align256(bytes); return p; };
    float *B0 = (float *)take((size_t)n * r * sizeof(float));
    float *T = (float *)take((size_t)r * r * sizeof(float));
    float *Z = (float *)take((size_t)n * r * sizeof(float));
    float *G = (float *)take((size_t)r * r * sizeof(float));
    uint32_t *Wimg = (uint32_t *)take(gemm3x_image_bytes(n, m));
    uint32_t *Vimg = (uint32_t *)take(gemm3x_image_bytes(r, m));
    uint32_t *Yimg = (uint32_t *)take(gemm3x_image_bytes(r, r));
    int *info = (int *)take(4 * sizeof(int));
    char *mw = take(msv);
    if (w) { w->B0 = B0; w->T = T; w->Z = Z; w->G = G; w->Wimg = Wimg; w->Vimg = Vimg; w->Yimg = Yimg; w->info = info; w->msvid = mw; w->msvid_bytes = msv; }
    *total = off;
    return MDBF_OK;
}
static mdbf_status_t check_shape(const char *who, int64_t n, int64_t m, int64_t r, int32_t l) {
    if (n < 1 || m < 1 || r < 1 || n > (1 << 21) || m > (1 << 21) || r > 32768 || n * r > (1LL << 31) - 1 || n * m > (1LL << 40)) {   // grid limits of the tiled kernels
        set_error("%s: sizes N=%lld M=%lld R=%lld outside the supported range", who, (long long)n, (long long)m, (long long)r);
        return MDBF_ERR_SHAPE;
    }
    if (r > n || r > m) {
        set_error("%s: the inner dimension R=%lld exceeds min(N, M) = min(%lld, %lld)", who, (long long)r, (long long)n, (long long)m);
        return MDBF_ERR_SHAPE;
    }
    if (l < 1 || l > kMaxL || l > n || l > r) {
        set_error("%s: l=%d outside [1, min(%d, N, R)]", who, l, kMaxL);
        return MDBF_ERR_SHAPE;
    }
    return MDBF_OK;
}

}  // namespace admm
}  // namespace mdbf

using namespace mdbf;

extern "C" mdbf_status_t mdbf_admm_workspace_bytes(int64_t n, int64_t m, int64_t r, int32_t l, size_t *bytes) {
    if (!bytes) { set_error("mdbf_admm_workspace_bytes: NULL pointer"); return MDBF_ERR_INVALID_ARG; }
    mdbf_status_t rc = admm::check_shape("mdbf_admm_workspace_bytes", n, m, r, l);
    if (rc) return rc;
    return admm::carve(nullptr, nullptr, n, m, r, l, bytes);
}

extern "C" mdbf_status_t mdbf_admm_factor_update(const float *W, int64_t w_rows, int64_t w_cols, int32_t transpose_w, const float *V,
                                                 int64_t r, float *U, float *Lambda, float rho, int32_t l, int32_t n_inner,
                                                 int32_t n_iter, const float *Q0, uint32_t *S_packed, float *Ul, float *Vl,
                                                 float *sigma, float *U_tilde, void *workspace, size_t workspace_bytes, void *stream) {
    const char *who = "mdbf_admm_factor_update";
    if (!W || !V || !U || !Lambda || !Q0 || !S_packed || !Ul || !Vl || !sigma || !workspace) {
        set_error("%s: NULL pointer", who);
        return MDBF_ERR_INVALID_ARG;
    }
    const int64_t n = transpose_w ? w_cols : w_rows, m = transpose_w ? w_rows : w_cols;
    mdbf_status_t rc = admm::check_shape(who, n, m, r, l);
    if (rc) return rc;
    if (!(rho > 0.f) || n_inner < 1 || n_inner > 1000 || n_iter < 1 || n_iter > 1000) {
        set_error("%s: rho=%g must be positive, n_inner=%d and n_iter=%d in [1, 1000]", who, (double)rho, n_inner, n_iter);
        return MDBF_ERR_INVALID_ARG;
    }
    admm::Scratch w;
    size_t need = 0;
    rc = admm::carve(&w, (char *)workspace, n, m, r, l, &need);
    if (rc) return rc;
    if (workspace_bytes < need || ((uintptr_t)workspace & 255u) != 0) {
        set_error("%s: the workspace must hold %zu bytes (mdbf_admm_workspace_bytes) on a 256-byte boundary; got %zu at %p", who, need,
                  workspace_bytes, workspace);
        return MDBF_ERR_INVALID_ARG;
    }
    int device = 0;
    rc = require_device(&device);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    admm::Libs *L = nullptr;
    rc = admm::get_libs(device, st, &L);
    if (rc) return rc;
    const int ni = (int)n, mi = (int)m, ri = (int)r;
    MDBF_CUDA(cudaMemsetAsync(w.info, 0, 4 * sizeof(int), st));
    // images: op(W)[i][k] = W[i * w_cols + k], or W[k * w_cols + i] when transposed;  V^T[j][k] = V[k * r + j]
    rc = gemm3x_split(V, 1, (size_t)r, ri, mi, w.Vimg, st);
    if (rc) return rc;
    // Fork.  Side stream: G = V^T V + rho I, its Cholesky factor L, Y = L^-T, G^-1 = Y Y^T as a product of Y's images with themselves - the inverse written out,
    // as Eq. admm-U-tilde has it, so that every inner iteration's solve is one product on the tensor cores instead of two
    // triangular solves with N right-hand sides on the FP32 pipe.  Caller's stream meanwhile: W's images and B0 = op(W) V,
    // on all SMs but a few that are left to the solver's small kernels.  Z is free until the loop below.
    cudaStream_t s2 = L->side;
    MDBF_CUDA(cudaEventRecord(L->fork, st));
    MDBF_CUDA(cudaStreamWaitEvent(s2, L->fork, 0));
    // the solver reads one triangle: half of V^T V; Y is triangular: a third of the products of Y Y^T
    rc = gemm3x_run(w.Vimg, w.Vimg, G3xOut{w.G, ri, false, nullptr, nullptr, G3X_UPPER}, ri, ri, mi, w.info + 2, s2);
    if (rc) return rc;
    admm::ridge_kernel<<<ceil_div(ri, 256), 256, 0, s2>>>(w.G, ri, rho);
    int lwork = 0;
    cusolverStatus_t ss = cusolverDnSpotrf_bufferSize(L->solver, CUBLAS_FILL_MODE_LOWER, ri, w.G, ri, &lwork);
    if (ss != CUSOLVER_STATUS_SUCCESS) { set_error("%s: cusolverDnSpotrf_bufferSize returned %d", who, (int)ss); return MDBF_ERR_CUDA; }
    rc = admm::grow_scratch(L, lwork, s2, who);
    if (rc) return rc;
    ss = cusolverDnSpotrf(L->solver, CUBLAS_FILL_MODE_LOWER, ri, w.G, ri, L->potrf_ws, L->potrf_floats, w.info);
    if (ss != CUSOLVER_STATUS_SUCCESS) { set_error("%s: cusolverDnSpotrf returned %d", who, (int)ss); return MDBF_ERR_CUDA; }
    // the solver's lower triangle is, read row-major, U = L^T; Y = U^-1 = L^-T.  Z is free until the loop, Y's images until Y is done
    rc = admm::tri_inverse(w.G, w.Z, w.T, w.Yimg, ri, w.info + 2, s2);
    if (rc) return rc;
    rc = gemm3x_split(w.Z, (size_t)r, 1, ri, ri, w.Yimg, s2);
    if (rc == MDBF_OK) rc = gemm3x_run(w.Yimg, w.Yimg, G3xOut{w.G, ri, false, nullptr, nullptr, G3X_FACTORS}, ri, ri, ri, w.info + 2, s2);
    if (rc) return rc;
    MDBF_CUDA(cudaEventRecord(L->join, s2));
    rc = transpose_w ? gemm3x_split(W, 1, (size_t)w_cols, ni, mi, w.Wimg, st) : gemm3x_split(W, (size_t)w_cols, 1, ni, mi, w.Wimg, st);
    if (rc == MDBF_OK) rc = gemm3x_run(w.Wimg, w.Vimg, w.B0, ni, ri, mi, w.info + 2, st, 24);
    if (rc) return rc;
    // Join; the inverse's images go where V's were (symmetric: rows serve as columns)
    MDBF_CUDA(cudaStreamWaitEvent(st, L->join, 0));
    rc = gemm3x_split(w.G, (size_t)r, 1, ri, ri, w.Vimg, st);
    if (rc) return rc;
    const int nwords = (int)((r + 31) / 32);
    for (int it = 0; it < n_inner; ++it) {
        // U_tilde = (B0 + rho (U - Lam)) G^-1 and Z = U_tilde + Lam: the right-hand side goes straight into images (where W's were) and U is
        // free from there on, so it takes U_tilde; the last one goes where the caller wants it.  Lam is added on the way out.
        rc = gemm3x_split_rhs(w.B0, U, Lambda, rho, ni, ri, w.Wimg, st);
        float *Ut = it == n_inner - 1 && U_tilde ? U_tilde : U;
        if (rc == MDBF_OK) rc = gemm3x_run(w.Wimg, w.Vimg, G3xOut{Ut, ri, false, Lambda, w.Z}, ni, ri, ri, w.info + 2, st);
        if (rc) return rc;
        rc = mdbf_msvid(w.Z, n, r, l, n_iter, Q0, S_packed, Ul, Vl, sigma, w.msvid, w.msvid_bytes, stream);
        if (rc) return rc;
        auto recon = l <= 4 ? admm::recon_dual_kernel<4> : l <= 8 ? admm::recon_dual_kernel<8> : l <= 16 ? admm::recon_dual_kernel<16> : admm::recon_dual_kernel<32>;
        recon<<<dim3(ceil_div(ri, admm::RC_COLS), ceil_div(ni, admm::RC_ROWS)), admm::RC_COLS, 0, st>>>(S_packed, Ul, Vl, l, Ut, U, Lambda, ni, ri, nwords);
    }
    admm::flag_kernel<<<1, 32, 0, st>>>(w.info, sigma, l);                      // the factorisation's flag or an expired wait
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}
