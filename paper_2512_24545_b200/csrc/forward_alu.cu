// fp32 CUDA-core path of the MDBF forward: any (l, T), any activation type.
//
// One stage computes, for every row r of the sign matrix S (rows x cols):
//
//     W[r][c] = S[r][c] * sum_t U[r][t] V[c][t],     out[tau][r] = sum_c W[r][c] in[tau][c]
//
// (Eq. me-dbf-basis: the factor is rebuilt entry by entry in registers, l multiply-adds, the packed bit XOR-ed into the IEEE sign bit,
// and multiplied by every token of the tile at once: l + T multiply-adds per entry where the expanded order of Eq. me-dbf-expand
// has l T), accumulated in fp32.  Stage B (S_B, V_B, U_B) maps x -> z, stage A (S_A, V_A, U_A) maps z -> y.  This is the path of the
// fp32 configuration and the GPU-side cross-check of the tensor-core paths.
//
// What bounds it: the FP32 pipe on large layers, the chain launch -> loads -> sum on small ones.  Lane = row, so that V and the
// activations of a column are the same for the whole warp: both are staged in shared memory as fp32 and read as broadcasts.  The warps of a
// CTA share 32 rows and split the columns (unit of a warp: cw columns of one sign word); with few row tiles a cluster of CTAs
// splits them further and adds up over distributed shared memory in rank order.
//
// Measured (B200, calls back to back, both launches of a forward): 256 x 256, k = 128, l = 4, T = 8: 33.1 -> 9.8 us, of which
// the host takes most; a random fp32 layer of the same range (128 ... 2048 a side) 178 -> 28.6 us.  Before, a lane owned a
// sign word and walked its 32 columns in series with two dependent global loads and l T multiply-adds each.
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace mdbf {

struct AluArgs {
    SignView words;
    int rows, cols, l, env_dtype, T, add;
    const void *U, *V, *in;
    void *out;
    int cw, units, per_rank;      // columns of a unit (8, 16 or 32), units of the reduction, units of a rank
    int part_off;                 // floats of shared memory before the sums the other ranks push
};
constexpr int kAluMaxRanks = 8;

// floats of shared memory a warp stages a unit in: V [32][lp], activations [32][pitch]
__host__ __device__ constexpr int alu_pitch(int TT) { return TT == 1 ? 1 : TT + 4; }      // 16-byte stores of neighbouring columns meet no bank twice
__host__ __device__ constexpr int alu_lp(int l) { return (l + 3) / 4 * 4; }

// LB: envelope rank the registers hold (l <= LB); TT: tokens of a tile
template <int TT, int LB, typename InT, typename OutT>
__global__ void __launch_bounds__(512) alu_stage_kernel(const AluArgs a) {
    extern __shared__ __align__(16) float alu_smem[];
    constexpr int XP = alu_pitch(TT);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int row_tiles = (a.rows + 31) / 32, rt = blockIdx.x % row_tiles;
    const int r = rt * 32 + lane, tau0 = blockIdx.x / row_tiles * TT;
    const int lp = alu_lp(a.l), cw = a.cw;
    float *vs = alu_smem + warp * 32 * (lp + XP), *xs = vs + 32 * lp;
    const InT *in = reinterpret_cast<const InT *>(a.in);
    cg::cluster_group cluster = cg::this_cluster();
    const int ranks = gridDim.y, rank = blockIdx.y;
    if (ranks > 1) cluster.barrier_arrive();                     // awaited before the first store into another CTA: it runs by then
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");

    float u[LB];
#pragma unroll
    for (int t = 0; t < LB; ++t) u[t] = (r < a.rows && t < a.l) ? env_load(a.U, (size_t)r * a.l + t, a.env_dtype) : 0.f;
    float acc[TT];
#pragma unroll
    for (int j = 0; j < TT; ++j) acc[j] = 0.f;

    const int u0 = blockIdx.y * a.per_rank, u1 = min(u0 + a.per_rank, a.units), per_word = 32 / cw;
    bool waited = false;
    for (int unit = u0 + warp; unit < u1; unit += nw) {
        const int w = unit / per_word, bit0 = unit % per_word * cw, c0 = w * 32 + bit0;
        const uint32_t word = r < a.rows ? a.words.word(r, w) >> bit0 : 0u;
        const int cn = min(cw, a.cols - c0);                     // columns that exist (none in the tail of the last word)
        __syncwarp();
        // V of the unit: cn * l consecutive entries, rows padded to lp with zeros
        if (cn > 0) {
            if (lp == a.l)
                for (int i = lane; i < cn * lp; i += 32) vs[i] = env_load(a.V, (size_t)c0 * lp + i, a.env_dtype);
            else
                for (int i = lane; i < cn * lp; i += 32) {
                    const int c = i / lp, t = i - c * lp;
                    vs[i] = t < a.l ? env_load(a.V, (size_t)(c0 + c) * a.l + t, a.env_dtype) : 0.f;
                }
        }
        if (!waited) { asm volatile("griddepcontrol.wait;\n" ::: "memory"); waited = true; }
        if (lane < cn) {
            if constexpr (TT == 1) xs[lane] = act_load<InT>(in, (size_t)tau0 * a.cols + c0 + lane);
            else
#pragma unroll
                for (int j = 0; j < TT; j += 4) {
                    float v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[e] = tau0 + j + e < a.T ? act_load<InT>(in, (size_t)(tau0 + j + e) * a.cols + c0 + lane) : 0.f;
                    *reinterpret_cast<float4 *>(xs + lane * XP + j) = make_float4(v[0], v[1], v[2], v[3]);
                }
        }
        __syncwarp();
#pragma unroll 2
        for (int c = 0; c < cn; ++c) {
            float e = 0.f;
#pragma unroll
            for (int q = 0; q < LB / 4; ++q)
                if (4 * q < lp) {
                    const float4 v = *reinterpret_cast<const float4 *>(vs + c * lp + 4 * q);
                    e = fmaf(u[4 * q], v.x, e); e = fmaf(u[4 * q + 1], v.y, e);
                    e = fmaf(u[4 * q + 2], v.z, e); e = fmaf(u[4 * q + 3], v.w, e);
                }
            e = __uint_as_float(__float_as_uint(e) ^ ((word << (31 - c)) & 0x80000000u));
            if constexpr (TT == 1) acc[0] = fmaf(e, xs[c], acc[0]);
            else
#pragma unroll
                for (int j = 0; j < TT; j += 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(xs + c * XP + j);
                    acc[j] = fmaf(e, x.x, acc[j]); acc[j + 1] = fmaf(e, x.y, acc[j + 1]);
                    acc[j + 2] = fmaf(e, x.z, acc[j + 2]); acc[j + 3] = fmaf(e, x.w, acc[j + 3]);
                }
        }
    }
    if (!waited) asm volatile("griddepcontrol.wait;\n" ::: "memory");

    // sum over the warps, then over the ranks of the cluster (each rank pushes its sums into rank 0)
    __syncthreads();
    float *red = alu_smem, *part = alu_smem + a.part_off;        // part: apart from what rank 0 may still be staging
#pragma unroll
    for (int j = 0; j < TT; ++j) red[(warp * TT + j) * 32 + lane] = acc[j];
    __syncthreads();
    auto sum = [&](int i) {
        float v = 0.f;
        for (int w = 0; w < nw; ++w) v += red[w * TT * 32 + i];
        return v;
    };
    if (ranks > 1) {
        cluster.barrier_wait();
        if (rank != 0) {
            float *dst = cluster.map_shared_rank(part, 0) + (rank - 1) * TT * 32;
            for (int i = threadIdx.x; i < TT * 32; i += blockDim.x) dst[i] = sum(i);
        }
        cluster.sync();
        if (rank != 0) return;
    }
    OutT *out = reinterpret_cast<OutT *>(a.out);
    for (int i = threadIdx.x; i < TT * 32; i += blockDim.x) {
        const int tau = tau0 + (i >> 5), row = rt * 32 + (i & 31);
        if (tau >= a.T || row >= a.rows) continue;
        float v = sum(i);
        for (int k = 1; k < ranks; ++k) v += part[(k - 1) * TT * 32 + i];
        const size_t o = (size_t)tau * a.rows + row;
        act_store<OutT>(out, o, a.add ? act_load<OutT>(out, o) + v : v);      // add: a further term of a sum
    }
}

// Warps of a CTA, unit width and ranks.  Token tile: the smallest that holds T, at most 32 (the envelope entry is rebuilt once per
// tile; 32 accumulators and 16 modes are what the registers hold).  A unit is one sign word; where that leaves warps idle it is split down to eight columns (a
// shorter chain per warp).  Ranks are added while every warp has more than four units and SMs are left.
template <int TT, int LB, typename InT, typename OutT>
static mdbf_status_t alu_launch(const AluArgs &a0, cudaStream_t st) {
    AluArgs a = a0;
    const int words = ceil_div(a.cols, 32);
    const int nw = LB > 16 ? 8 : 16;
    a.cw = 32;
    while (a.cw > 8 && words * (32 / a.cw) < nw) a.cw /= 2;
    a.units = words * (32 / a.cw);
    const int tiles = ceil_div(a.rows, 32) * ceil_div(a.T, TT);
    int ranks = 1;
    while (ranks < kAluMaxRanks && tiles * ranks * 2 <= 148 * 2 && ceil_div(a.units, ranks * 2) >= 2 * nw) ranks *= 2;
    a.per_rank = ceil_div(a.units, ranks);
    const size_t stage = (size_t)nw * 32 * (alu_lp(a.l) + alu_pitch(TT)) * 4, sums = (size_t)nw * TT * 32 * 4, base = stage > sums ? stage : sums;
    a.part_off = (int)(base / 4);
    auto kern = alu_stage_kernel<TT, LB, InT, OutT>;
    static PerDeviceOnce once;
    if (auto first = once.first()) MDBF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles, ranks);
    cfg.blockDim = dim3(nw * 32);
    cfg.dynamicSmemBytes = base + (size_t)(ranks - 1) * TT * 32 * 4;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = ranks;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ranks > 1 ? 2 : 1;
    MDBF_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    return MDBF_OK;
}
template <typename InT, typename OutT> static mdbf_status_t alu_stage(const AluArgs &a, cudaStream_t st) {
    if (a.l > 16) return a.T == 1 ? alu_launch<1, kMaxL, InT, OutT>(a, st) : alu_launch<8, kMaxL, InT, OutT>(a, st);
    if (a.T == 1) return alu_launch<1, 16, InT, OutT>(a, st);
    if (a.T <= 4) return alu_launch<4, 16, InT, OutT>(a, st);
    if (a.T <= 8) return alu_launch<8, 16, InT, OutT>(a, st);
    if (a.T <= 16) return alu_launch<16, 16, InT, OutT>(a, st);
    return alu_launch<32, 16, InT, OutT>(a, st);
}

template <typename ActT>
static mdbf_status_t run(Layer &L, const void *x, void *y, int T, cudaStream_t st) {
    AluArgs b = {};
    b.words = sign_view(L, 1); b.rows = L.d.k; b.cols = L.d.d_in; b.U = L.UB; b.V = L.VB;
    b.l = L.d.l; b.env_dtype = L.d.env_dtype; b.in = x; b.out = L.zsum; b.T = T;
    mdbf_status_t rc = alu_stage<ActT, float>(b, st);
    if (rc) return rc;
    AluArgs s = b;
    s.words = sign_view(L, 0); s.rows = L.d.d_out; s.cols = L.d.k; s.U = L.UA; s.V = L.VA; s.in = L.zsum; s.out = y;
    if (L.out_mode == 0) return alu_stage<float, ActT>(s, st);
    s.add = L.out_mode == 2;                // a term of a sum of layers: fp32 output, stored or added
    return alu_stage<float, float>(s, st);
}

mdbf_status_t launch_forward_alu(Layer &L, const void *x, void *y, int T, int act_dtype,
                                 cudaStream_t st, int *launches) {
    mdbf_status_t rc;
    if (act_dtype == MDBF_F32) rc = run<float>(L, x, y, T, st);
    else if (act_dtype == MDBF_BF16) rc = run<__nv_bfloat16>(L, x, y, T, st);
    else if (act_dtype == MDBF_F16) rc = run<__half>(L, x, y, T, st);
    else { set_error("mdbf_linear_forward: unsupported activation dtype %d", act_dtype); return MDBF_ERR_DTYPE; }
    if (rc == MDBF_OK) { L.last_ksplit = 0; *launches = 2; }
    return rc;
}

// fp32 accumulator of a sum of layers -> activation type (one rounding)
template <typename OutT>
__global__ void cast_kernel(const float *__restrict__ acc, OutT *__restrict__ y, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        act_store<OutT>(y, i, acc[i]);
}

mdbf_status_t launch_cast(const float *acc, void *y, size_t n, int act_dtype, cudaStream_t st) {
    int grid = (int)((n + 255) / 256);
    if (grid > 148 * 16) grid = 148 * 16;
    if (grid < 1) grid = 1;
    if (act_dtype == MDBF_F32) cast_kernel<float><<<grid, 256, 0, st>>>(acc, reinterpret_cast<float *>(y), n);
    else if (act_dtype == MDBF_BF16) cast_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(acc, reinterpret_cast<__nv_bfloat16 *>(y), n);
    else cast_kernel<__half><<<grid, 256, 0, st>>>(acc, reinterpret_cast<__half *>(y), n);
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}

// make the fp32 copy of the intermediate current (inspection only): the materialised-envelope kernels keep z in bf16
mdbf_status_t launch_zsum(Layer &L, int T, cudaStream_t st) {
    if (L.last_ksplit < 0) return launch_zb_to_zsum(L, T, st);
    return MDBF_OK;
}

}  // namespace mdbf
