// Dense fp32 product C = A B on the tensor cores at close to fp32 accuracy: tcgen05 kind::f16 on a scaled two-part split
//     a b  ~  a_hi b_hi + 2^-11 (a_hi b_lo + a_lo b_hi)  (the dropped product of the low parts is below 2^-24 a b)
// with fp32 accumulation in tensor memory.  It serves the least-squares step of the ADMM refinement (W V and V^T V,
// Eq. admm-U-tilde), where the FP32 pipe would need eight times as long.
//
// The split.  A row of an operand (a row of A, a column of B) is multiplied by the power of two that brings its largest entry into
// [2^14, 2^15); hi = the scaled entry rounded to fp16, lo = 2^11 times the exact residual, rounded to fp16.  With the factor lo keeps the
// exponent of hi, so entries down to 2^-29 of the row's largest have 11 + 11 significant bits, the same as two TF32 parts, and smaller ones
// an absolute error of 2^-51 of it (without the factor: 2^-17 and 2^-40, which shows where small entries of W meet large ones of V; rows and
// columns scaled against each other by 10^+-4: 6.0e-5 of the iterate without it, 7.9e-7 with it, 2.5e-6 with TF32 parts).  The cross terms
// of a K block are formed first, and the first product of the high parts scales the accumulator by 2^-11 as it adds to it.  C is multiplied by
// both inverse scales on the way out (exact).  fp16 operands issue at twice the TF32 rate and are half the bytes: 8192 x 3712 x 3712
// 943 -> 566 us, 8192 x 3712 x 8192 on 124 SMs 2193 -> 1271, with single accumulations over two K blocks; the factor and one K block per
// accumulation take 2.5 % more.  Error of an ADMM iterate against fp64 at that size: TF32 2.0e-6, without the factor 1.4e-6, now 5.8e-7.
//
// Two passes.  The split kernels turn an operand into "images": per tile of 128 rows (output rows for A, output
// columns for B) and block of 64 contraction indices one 32 KB piece holding hi (128 rows of 64 fp16 values, 128 bytes
// each) and lo (the same shape behind it), rows K-major with the 128B swizzle a shared-memory matrix descriptor expects
// (16-byte chunk c of row r at position c ^ (r & 7)); tails are zero.  Behind the pieces lie the rows' inverse scales, behind those the
// bits of their largest magnitudes.  Either operand may be given transposed: an
// element is read at src[i * stride_i + k * stride_k] with one of the strides equal to one.
// gemm3x_kernel: one CTA per SM walks over 128 x 256 tiles of C (two column tiles of B side by side: the stream from L2
// into shared memory, 96 KB per K block, is what bounds the kernel, and a wider tile spends less of it per flop); one
// lane streams the pieces of each K block into a ring by bulk copies, one warp issues  D = A_hi B_lo, D += A_lo B_hi,
// D = 2^-11 D + A_hi B_hi  (N = 256, four K steps of 16 each), the eight epilogue warps add the K blocks' accumulators up and store.  Every wait is bounded; on expiry the status word is
// set and the tiles still to be written come out as NaN.
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "tmem_ptx.cuh"

namespace mdbf {
namespace g3x {

constexpr int TILE = 128, KB = 64;
constexpr int HALF = TILE * KB * 2;            // bytes of the hi (or lo) part of a piece
constexpr int PIECE = 2 * HALF;                // 32 KB
constexpr int STAGES = 2;
constexpr int LO_SHIFT = 11;                   // lo is the residual times 2^11
constexpr int STAGE_BYTES = 3 * PIECE;         // A piece, then B_hi of two column tiles, then their B_lo
constexpr int EPI_WARPS = 8;                   // two per quarter of the TMEM lanes, each with half of the tile's columns
constexpr int THREADS = (EPI_WARPS + 2) * 32;  // epilogue warps, loader, issuer
constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE_BYTES;

// scale and inverse scale of a row from the bits of its largest magnitude: powers of two, 2^14 <= max * scale < 2^15 (an all-zero or
// denormal row is scaled up as far as the inverse stays normal, a row with an infinity or NaN not at all)
__device__ __forceinline__ float row_scale(uint32_t maxbits, float *inverse) {
    const int e = (int)(maxbits >> 23);
    const int f = e == 255 ? 127 : min(253, 268 - e);
    *inverse = __uint_as_float((uint32_t)(254 - f) << 23);
    return __uint_as_float((uint32_t)f << 23);
}
// eight entries -> 16 bytes of hi and 16 of lo
__device__ __forceinline__ void split8(const float (&v)[8], float scale, uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float a = v[2 * u] * scale, b = v[2 * u + 1] * scale;
        const __half2 hh = __floats2half2_rn(a, b);
        const float2 back = __half22float2(hh);
        const __half2 ll = __floats2half2_rn((a - back.x) * (float)(1 << LO_SHIFT), (b - back.y) * (float)(1 << LO_SHIFT));
        h[u] = *reinterpret_cast<const uint32_t *>(&hh);
        l[u] = *reinterpret_cast<const uint32_t *>(&ll);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ void store_split(unsigned char *piece, int r, int chunk, const uint4 &hi, const uint4 &lo) {
    const int off = r * 128 + ((chunk ^ (r & 7)) << 4);
    *reinterpret_cast<uint4 *>(piece + off) = hi;
    *reinterpret_cast<uint4 *>(piece + HALF + off) = lo;
}
// What a row is read from: a matrix, or the right-hand side of the refinement's system, B0 + rho (U - Lam) (Eq. admm-U-tilde), which
// this way is never written out.
struct RowsOf {
    const float *src;
    __device__ __forceinline__ bool vec(size_t at) const { return (reinterpret_cast<uintptr_t>(src + at) & 15u) == 0; }
    __device__ __forceinline__ float at(size_t e) const { return src[e]; }
    __device__ __forceinline__ float4 at4(size_t e) const { return *reinterpret_cast<const float4 *>(src + e); }
};
struct RowsOfRhs {
    const float *b0, *u, *lam;
    float rho;
    __device__ __forceinline__ bool vec(size_t at) const {
        return ((reinterpret_cast<uintptr_t>(b0 + at) | reinterpret_cast<uintptr_t>(u + at) | reinterpret_cast<uintptr_t>(lam + at)) & 15u) == 0;
    }
    __device__ __forceinline__ float at(size_t e) const { return b0[e] + rho * (u[e] - lam[e]); }
    __device__ __forceinline__ float4 at4(size_t e) const {
        const float4 b = *reinterpret_cast<const float4 *>(b0 + e), x = *reinterpret_cast<const float4 *>(u + e), y = *reinterpret_cast<const float4 *>(lam + e);
        return make_float4(b.x + rho * (x.x - y.x), b.y + rho * (x.y - y.y), b.z + rho * (x.z - y.z), b.w + rho * (x.w - y.w));
    }
};
// Contraction indices contiguous: CTA = row, NV chunks of eight entries per thread stay in registers between the search for the largest
// magnitude and the split, so that the source is read once (what a longer row has beyond them is read twice); eight lanes write a
// row's 128 bytes of a K block.
// Bound by memory: the right-hand side of 8192 x 3712 in 67 us (16 bytes per entry, 7.3 TB/s with what L2 still holds), 87 + 60 us as a
// pass of its own and a split that read its row twice.
template <class SRC, int NV>
__global__ void __launch_bounds__(256) split_rows_kernel(const SRC src, size_t stride_i, int ni, int nk, int nkb,
                                                         unsigned char *__restrict__ img, float *__restrict__ inv) {
    __shared__ float warp_max[8];
    const int row = blockIdx.x, tid = threadIdx.x;
    const size_t base = (size_t)min(row, ni - 1) * stride_i;
    const int n = row < ni ? nk : 0;                             // rows behind the matrix are zeros
    const bool vec = src.vec(base);
    auto load = [&](int chunk, float (&v)[8]) {
        const int k0 = 8 * chunk;
        if (vec && k0 + 8 <= n) {
            const float4 x = src.at4(base + k0), y = src.at4(base + k0 + 4);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = k0 + u < n ? src.at(base + k0 + u) : 0.f;
        }
    };
    float v[NV][8], m = 0.f;
#pragma unroll
    for (int c = 0; c < NV; ++c) load(tid + 256 * c, v[c]);
#pragma unroll
    for (int c = 0; c < NV; ++c)
#pragma unroll
        for (int u = 0; u < 8; ++u) m = fmaxf(m, fabsf(v[c][u]));
    for (int chunk = tid + 256 * NV; 8 * chunk < n; chunk += 256) {
        float x[8];
        load(chunk, x);
#pragma unroll
        for (int u = 0; u < 8; ++u) m = fmaxf(m, fabsf(x[u]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) warp_max[tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, warp_max[w]);
    float inverse;
    const float scale = row_scale(__float_as_uint(m), &inverse);
    if (tid == 0) inv[row] = inverse;
    unsigned char *tile = img + (size_t)(row / TILE) * nkb * PIECE;
    const int r = row % TILE;
    auto store = [&](int chunk, const float (&x)[8]) {
        uint4 hi, lo;
        split8(x, scale, hi, lo);
        store_split(tile + (size_t)(chunk >> 3) * PIECE, r, chunk & 7, hi, lo);
    };
#pragma unroll
    for (int c = 0; c < NV; ++c)
        if (tid + 256 * c < 8 * nkb) store(tid + 256 * c, v[c]);
    for (int chunk = tid + 256 * NV; chunk < 8 * nkb; chunk += 256) {
        float x[8];
        load(chunk, x);
        store(chunk, x);
    }
}
template <class SRC>
static void launch_split_rows(const SRC &src, size_t stride_i, int rows, int depth, int nkb, int tiles, unsigned char *pieces, float *inv, cudaStream_t st) {
    const int grid = tiles * TILE;
    if (nkb <= 32) split_rows_kernel<SRC, 1><<<grid, 256, 0, st>>>(src, stride_i, rows, depth, nkb, pieces, inv);
    else if (nkb <= 64) split_rows_kernel<SRC, 2><<<grid, 256, 0, st>>>(src, stride_i, rows, depth, nkb, pieces, inv);
    else split_rows_kernel<SRC, 4><<<grid, 256, 0, st>>>(src, stride_i, rows, depth, nkb, pieces, inv);
}
// Rows contiguous (a transposed operand): largest magnitudes by a pass of their own, thread = row, CM_DEPTH contraction indices per CTA, all of
// its loads in flight (1024 x 1024: 22 us with 256 indices per CTA, sixteen CTAs, eight loads at a time) ...
constexpr int CM_DEPTH = 32;
__global__ void __launch_bounds__(256) column_max_kernel(const float *__restrict__ src, size_t stride_k, int ni, int nk, uint32_t *__restrict__ maxbits) {
    const int i = blockIdx.y * 256 + threadIdx.x, k0 = blockIdx.x * CM_DEPTH;
    if (i >= ni) return;
    float m = 0.f;
#pragma unroll
    for (int u = 0; u < CM_DEPTH; ++u) m = fmaxf(m, fabsf(src[(size_t)min(k0 + u, nk - 1) * stride_k + i]));
    atomicMax(maxbits + i, __float_as_uint(m));                  // magnitudes order like their bits
}
// ... then the images, thread = row (consecutive rows are consecutive in memory), two threads per row share its 8 chunks
__global__ void __launch_bounds__(256) split_columns_kernel(const float *__restrict__ src, size_t stride_k, int ni, int nk, int nkb,
                                                            unsigned char *__restrict__ img, float *__restrict__ inv, const uint32_t *__restrict__ maxbits) {
    const int kb = blockIdx.x, it = blockIdx.y;
    unsigned char *piece = img + ((size_t)it * nkb + kb) * PIECE;
    const int r = threadIdx.x & 127, i = it * TILE + r;
    float inverse;
    const float scale = row_scale(maxbits[i], &inverse);         // (zero behind the matrix)
    if (kb == 0 && threadIdx.x < TILE) inv[i] = inverse;
#pragma unroll
    for (int chunk = threadIdx.x >> 7; chunk < 8; chunk += 2) {
        const int k0 = kb * KB + 8 * chunk;
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = (i < ni && k0 + u < nk) ? src[(size_t)i + (size_t)(k0 + u) * stride_k] : 0.f;
        uint4 hi, lo;
        split8(v, scale, hi, lo);
        store_split(piece, r, chunk, hi, lo);
    }
}

// Tile t of the walk: row tile by row tile; of a symmetric result only the tiles that reach the diagonal or lie above it.
__device__ __forceinline__ void tile_of(int t, int ntn2, int part, int &mt, int &nt2) {
    if (part != G3X_UPPER) {
        mt = t / ntn2;
        nt2 = t - mt * ntn2;
        return;
    }
    int p = 0;                                                   // row tiles 2p and 2p + 1 start at column tile p
    while (t >= 2 * (ntn2 - p)) { t -= 2 * (ntn2 - p); ++p; }
    const int second = t >= ntn2 - p;
    mt = 2 * p + second;
    nt2 = p + t - (second ? ntn2 - p : 0);
}
// first K block with anything in it: rows of upper triangular operands are zero before the diagonal
__device__ __forceinline__ int first_kb(int part, int mt, int nt2) { return part == G3X_FACTORS ? max(mt * TILE, nt2 * 2 * TILE) / KB : 0; }

// Persistent: CTA c takes the tiles c, c + gridDim.x, ... (row tile = t / ntn2, so that CTAs running side by side share
// their pieces of A in L2).  Two accumulators of 256 tensor-memory columns alternate: the epilogue of
// one K block runs under the products of the next.  All three terms of a K block accumulate into the same columns, and the K blocks'
// sums are added in fp32 by the epilogue, in registers: the tensor core's accumulation is not rounded to nearest, and its one-sided error
// grows with the number of accumulations (6e-5 of the result over 8192 contraction indices, measured).  ntn is
// the number of 128-column tiles of B's images, ntn2 = ceil(ntn / 2) the number of tiles here; an odd last tile has no
// second half: nothing is copied for it, the products read whatever the buffer holds, and nothing of it is stored.
__global__ void __launch_bounds__(THREADS, 1) gemm3x_kernel(const uint32_t *__restrict__ Aimg, const uint32_t *__restrict__ Bimg,
                                                            const float *__restrict__ Ainv, const float *__restrict__ Binv, const G3xOut o, int n, int r, int nkb, int ntn, int ntn2, int ntiles,
                                                            int32_t *__restrict__ status) {
    using namespace tm;
    extern __shared__ unsigned char g3_smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * STAGES + 4];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag_s;
    volatile int *abort_flag = &abort_flag_s;
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const uint32_t smem_base = (smem_u32(g3_smem_raw) + 1023u) & ~1023u;
    const uint32_t full_bar = smem_u32(&bars[0]), empty_bar = smem_u32(&bars[STAGES]);
    const uint32_t acc_full = smem_u32(&bars[2 * STAGES]), acc_empty = smem_u32(&bars[2 * STAGES + 2]);
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar + 8 * s, 1);                      // the loader's expect_tx
            mbar_init(empty_bar + 8 * s, 1);                     // the issuer's commit
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(acc_full + 8 * a, 1);                      // the issuer's commit after a tile's last K block
            mbar_init(acc_empty + 8 * a, EPI_WARPS * 32);        // every epilogue thread, once it has read its part
        }
        abort_flag_s = 0;
        fence_barrier_init();
    }
    if (warp == EPI_WARPS + 1) {
        tmem_alloc(smem_u32(&tmem_base_slot), 512u);             // two accumulators of 256 columns; one CTA per SM
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(tmem_base_slot);

    if (warp < EPI_WARPS) {
        // ===================================== epilogue =====================================
        // thread = one row and one half (128 columns) of the tile; the K blocks' sums are added in registers, in fp32
        const int half = warp >> 2;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const bool vec = (o.ldc & 3) == 0 && ((reinterpret_cast<uintptr_t>(o.C) | reinterpret_cast<uintptr_t>(o.add) | reinterpret_cast<uintptr_t>(o.sum)) & 15u) == 0;
        bool alive = true;
        int it = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            int mt, nt2;
            tile_of(t, ntn2, o.part, mt, nt2);
            const int nk = nkb - first_kb(o.part, mt, nt2), nch = max(nk, 1);
            const int row = mt * TILE + (warp & 3) * 32 + lane;
            const int col0 = nt2 * 2 * TILE + half * TILE;
            float sum[TILE];
            for (int ch = 0; ch < nch; ++ch, ++it) {
                const int as = it & 1;
                if (alive) alive = mbar_wait(acc_full + 8 * as, ((uint32_t)(it >> 1)) & 1u, abort_flag, status);
                alive = __all_sync(0xffffffffu, alive);
                tc_fence_after();
                if (alive && nk > 0) {
#pragma unroll
                    for (int j = 0; j < TILE / 16; ++j) {
                        uint32_t d[16];
                        tmem_ld16(tmem + lane_base + (uint32_t)(as * 2 * TILE + half * TILE + 16 * j), d);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[16 * j + e] = ch == 0 ? __uint_as_float(d[e]) : sum[16 * j + e] + __uint_as_float(d[e]);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < TILE; ++e) sum[e] = alive ? 0.f : __int_as_float(0x7fc00000);
                }
                tc_fence_before();
                if (alive) mbar_arrive(acc_empty + 8 * as);       // the accumulator may be overwritten
            }
            if (row < n && col0 < r) {
                const size_t at = (size_t)row * o.ldc + col0;
                const float ri = Ainv[row], sign = o.negate ? -1.f : 1.f;
                // both inverse scales, the smaller one first: a large row times a small column stays inside fp32 on the way
                auto scaled = [&](float v, float ci) { return v * (fminf(ri, ci) * sign) * fmaxf(ri, ci); };
                if (vec && col0 + TILE <= r) {
#pragma unroll
                    for (int e0 = 0; e0 < TILE; e0 += 32) {      // eight loads of the addend in flight: 8192 x 3712, 566 us without it: +30, +85 one at a time
                        float4 a[8];
                        if (o.sum) {
#pragma unroll
                            for (int q = 0; q < 8; ++q) a[q] = *reinterpret_cast<const float4 *>(o.add + at + e0 + 4 * q);
                        }
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int e = e0 + 4 * q;
                            const float4 ci = *reinterpret_cast<const float4 *>(Binv + col0 + e);
                            const float4 v = make_float4(scaled(sum[e], ci.x), scaled(sum[e + 1], ci.y), scaled(sum[e + 2], ci.z), scaled(sum[e + 3], ci.w));
                            if (o.C) *reinterpret_cast<float4 *>(o.C + at + e) = v;
                            if (o.sum) *reinterpret_cast<float4 *>(o.sum + at + e) = make_float4(v.x + a[q].x, v.y + a[q].y, v.z + a[q].z, v.w + a[q].w);
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < TILE; ++e)
                        if (col0 + e < r) {
                            const float v = scaled(sum[e], Binv[col0 + e]);
                            if (o.C) o.C[at + e] = v;
                            if (o.sum) o.sum[at + e] = v + o.add[at + e];
                        }
                }
            }
        }
    } else if (warp == EPI_WARPS) {
        // ====================================== loader ======================================
        if (lane == 0) {
            bool alive = true;
            int g = 0;                                           // K blocks issued so far, over all of this CTA's tiles
            for (int t = blockIdx.x; t < ntiles && alive; t += gridDim.x) {
                int mt, nt2;
                tile_of(t, ntn2, o.part, mt, nt2);
                const bool two = 2 * nt2 + 1 < ntn;              // the tile has a second column tile
                const uint32_t *a_src = Aimg + (size_t)mt * nkb * (PIECE / 4);
                const uint32_t *b0_src = Bimg + (size_t)(2 * nt2) * nkb * (PIECE / 4), *b1_src = b0_src + (size_t)nkb * (PIECE / 4);
                for (int kb = first_kb(o.part, mt, nt2); kb < nkb && alive; ++kb, ++g) {
                    const int s = g % STAGES;
                    alive = mbar_wait(empty_bar + 8 * s, (((uint32_t)(g / STAGES)) & 1u) ^ 1u, abort_flag, status);
                    if (!alive) break;
                    const uint32_t dst = smem_base + (uint32_t)(s * STAGE_BYTES);
                    mbar_arrive_expect_tx(full_bar + 8 * s, (uint32_t)(two ? 3 * PIECE : 2 * PIECE));
                    bulk_load(dst, a_src + (size_t)kb * (PIECE / 4), (uint32_t)PIECE, full_bar + 8 * s);
                    const uint32_t *b0 = b0_src + (size_t)kb * (PIECE / 4), *b1 = b1_src + (size_t)kb * (PIECE / 4);
                    bulk_load(dst + (uint32_t)PIECE, b0, (uint32_t)HALF, full_bar + 8 * s);                          // B_hi, first 128 rows
                    bulk_load(dst + (uint32_t)(2 * PIECE), b0 + HALF / 4, (uint32_t)HALF, full_bar + 8 * s);         // B_lo, first 128 rows
                    if (two) {
                        bulk_load(dst + (uint32_t)(PIECE + HALF), b1, (uint32_t)HALF, full_bar + 8 * s);             // B_hi, rows 128..255
                        bulk_load(dst + (uint32_t)(2 * PIECE + HALF), b1 + HALF / 4, (uint32_t)HALF, full_bar + 8 * s);
                    }
                }
            }
        }
        __syncwarp();
    } else {
        // ====================================== issuer ======================================
        const uint32_t idesc = make_idesc_fmt(2 * TILE, 0u);
        bool alive = true;
        int s = 0, it = 0;
        uint32_t ph = 0;
        for (int t = blockIdx.x; t < ntiles && alive; t += gridDim.x) {
            int mt, nt2;
            tile_of(t, ntn2, o.part, mt, nt2);
            const int nk = nkb - first_kb(o.part, mt, nt2), nch = max(nk, 1);
            for (int ch = 0; ch < nch && alive; ++ch, ++it) {
                const int as = it & 1;
                alive = __all_sync(0xffffffffu, mbar_wait(acc_empty + 8 * as, (((uint32_t)(it >> 1)) & 1u) ^ 1u, abort_flag, status));
                if (!alive) break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(as * 2 * TILE);
                if (nk > 0) {                                    // one K block
                    alive = __all_sync(0xffffffffu, mbar_wait(full_bar + 8 * s, ph, abort_flag, status));
                    tc_fence_after();
                    const uint32_t stage = smem_base + (uint32_t)(s * STAGE_BYTES);
                    const uint64_t a_hi = make_smem_desc(stage), a_lo = make_smem_desc(stage + (uint32_t)HALF);
                    const uint64_t b_hi = make_smem_desc(stage + (uint32_t)PIECE), b_lo = make_smem_desc(stage + (uint32_t)(2 * PIECE));
                    if (alive && elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)           // 16 fp16 = 32 bytes per K step; the first one clears the accumulator
                            umma_ss(d, a_hi + (uint64_t)(2 * ks), b_lo + (uint64_t)(2 * ks), idesc, ks > 0 ? 1u : 0u);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) umma_ss(d, a_lo + (uint64_t)(2 * ks), b_hi + (uint64_t)(2 * ks), idesc, 1u);
                        umma_ss_rescale<LO_SHIFT>(d, a_hi, b_hi, idesc);
#pragma unroll
                        for (int ks = 1; ks < 4; ++ks) umma_ss(d, a_hi + (uint64_t)(2 * ks), b_hi + (uint64_t)(2 * ks), idesc, 1u);
                        umma_commit(empty_bar + 8 * s);
                    }
                    __syncwarp();
                    if (++s == STAGES) { s = 0; ph ^= 1u; }
                }
                if (elect_one()) {
                    if (alive && nk > 0) umma_commit(acc_full + 8 * as);
                    else mbar_arrive(acc_full + 8 * as);
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) drain_delay();                              // let copies in flight land before the shared memory goes back
    if (warp == EPI_WARPS + 1) tmem_dealloc(tmem, 512u);
}

}  // namespace g3x

// pieces, then per tile row the inverse scale and the bits of the largest magnitude
static size_t g3x_pieces(int rows, int depth) { return (size_t)ceil_div(rows, g3x::TILE) * (size_t)ceil_div(depth, g3x::KB) * g3x::PIECE; }
size_t gemm3x_image_bytes(int64_t rows, int64_t depth) {
    return g3x_pieces((int)rows, (int)depth) + (size_t)ceil_div((int)rows, g3x::TILE) * g3x::TILE * 8;
}
static float *g3x_inverse(uint32_t *img, int rows, int depth) { return reinterpret_cast<float *>(reinterpret_cast<char *>(img) + g3x_pieces(rows, depth)); }

// images of an operand with `rows` tile rows and `depth` contraction indices; element (i, k) at src[i * stride_i + k * stride_k]
mdbf_status_t gemm3x_split(const float *src, size_t stride_i, size_t stride_k, int rows, int depth, uint32_t *img, cudaStream_t st) {
    const int nkb = ceil_div(depth, g3x::KB), tiles = ceil_div(rows, g3x::TILE);
    float *inv = g3x_inverse(img, rows, depth);
    unsigned char *pieces = reinterpret_cast<unsigned char *>(img);
    if (stride_k == 1) {
        g3x::launch_split_rows(g3x::RowsOf{src}, stride_i, rows, depth, nkb, tiles, pieces, inv, st);
    } else if (stride_i == 1) {
        uint32_t *maxbits = reinterpret_cast<uint32_t *>(inv + (size_t)tiles * g3x::TILE);
        MDBF_CUDA(cudaMemsetAsync(maxbits, 0, (size_t)tiles * g3x::TILE * 4, st));
        g3x::column_max_kernel<<<dim3(ceil_div(depth, g3x::CM_DEPTH), ceil_div(rows, 256)), 256, 0, st>>>(src, stride_k, rows, depth, maxbits);
        g3x::split_columns_kernel<<<dim3(nkb, tiles), 256, 0, st>>>(src, stride_k, rows, depth, nkb, pieces, inv, maxbits);
    } else { set_error("gemm3x_split: one of the strides must be 1"); return MDBF_ERR_INVALID_ARG; }
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}

mdbf_status_t gemm3x_split_rhs(const float *B0, const float *U, const float *Lam, float rho, int rows, int depth, uint32_t *img, cudaStream_t st) {
    g3x::launch_split_rows(g3x::RowsOfRhs{B0, U, Lam, rho}, (size_t)depth, rows, depth, ceil_div(depth, g3x::KB), ceil_div(rows, g3x::TILE),
                           reinterpret_cast<unsigned char *>(img), g3x_inverse(img, rows, depth), st);
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}

// C (n x r, row-major) = A B from the operands' images (A: n rows, B: r rows, both `depth` deep); spare_sms SMs are left
// to kernels of another stream
mdbf_status_t gemm3x_run(const uint32_t *Aimg, const uint32_t *Bimg, float *C, int n, int r, int depth, int32_t *status, cudaStream_t st,
                         int spare_sms) {
    const G3xOut o = {C, r, false, nullptr, nullptr, G3X_ALL};
    return gemm3x_run(Aimg, Bimg, o, n, r, depth, status, st, spare_sms);
}
mdbf_status_t gemm3x_run(const uint32_t *Aimg, const uint32_t *Bimg, const G3xOut &o, int n, int r, int depth, int32_t *status, cudaStream_t st,
                         int spare_sms) {
    static PerDeviceOnce once;
    if (auto first = once.first()) MDBF_CUDA(cudaFuncSetAttribute(g3x::gemm3x_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g3x::SMEM));
    const int ntm = ceil_div(n, g3x::TILE), ntn = ceil_div(r, g3x::TILE);
    int sms = 0;
    mdbf_status_t rc = device_sms(&sms);
    if (rc) return rc;
    const int ntn2 = ceil_div(ntn, 2);
    if (o.part != G3X_ALL && (n != r || (o.part == G3X_FACTORS && depth != n))) { set_error("gemm3x_run: a symmetric result is square"); return MDBF_ERR_INVALID_ARG; }
    int ntiles = ntm * ntn2;
    if (o.part == G3X_UPPER) {
        ntiles = 0;
        for (int mt = 0; mt < ntm; ++mt) ntiles += ntn2 - mt / 2;
    }
    g3x::gemm3x_kernel<<<std::min(ntiles, std::max(1, sms - spare_sms)), g3x::THREADS, g3x::SMEM, st>>>(
        Aimg, Bimg, g3x_inverse(const_cast<uint32_t *>(Aimg), n, depth), g3x_inverse(const_cast<uint32_t *>(Bimg), r, depth), o, n, r,
        ceil_div(depth, g3x::KB), ntn, ntn2, ntiles, status);
    MDBF_CUDA(cudaGetLastError());
    return MDBF_OK;
}

}  // namespace mdbf
