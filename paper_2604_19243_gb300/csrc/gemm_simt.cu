// SIMT (CUDA-core) form of the gathered GEMM of gemm_common.cuh, in FP32 or FP64: the FMM_FP32 and
// FMM_FP64 contractions (but the M2L where gemm_f16.cu and gemm_f64.cu take it) and the leaf closing of
// every mode.
//
// A CTA of 128 threads computes 64 rows x 64 columns (FP64: 32), 4 x 8 (4 x 4) a thread.  Rows and
// operators go to shared memory as they lie in global memory (K contiguous), 64 bytes of K a stage, by
// 16-byte cp.async three stages ahead, one barrier a stage; the chunks of all segments form one
// sequence, so that the copies run on across segments.  The shared rows are 80 bytes apart: the rows
// that the lanes of a warp read together then lie on different banks.  Every output is one sequence of
// fused multiply-adds in the order of K and of the segments.
//
// What bounds it: the FMA pipe on many rows (FP64: 0.9 of 1.25 TFLOP/s); on the few rows of the coarse
// levels the latency of a stage.  Against 64 x 32 tiles of 4 x 4 outputs a thread with loads and
// products in turn, one GB300, p = 6, FP32: U2U into 512 parents 354 -> 54 us and into 4096 parents 355
// -> 84 us; the two closing products of 32,768 leaves 200 -> 118 us; 64 columns instead of 32 for FP64
// would cost 28% (192 columns for 160).
#include <algorithm>

#include "gemm_common.cuh"
#include "tcgen05.cuh"

namespace fmm {
namespace {

constexpr int BM = 64, THREADS = 128;
template <typename T> constexpr int kCols = sizeof(T) == 8 ? 32 : 64;   // columns per CTA
constexpr int kStages = 4;
constexpr int kPitch = 80;                        // bytes of a shared row: 64 of K and a pad

// one output: the products of 16 bytes of K added in order
__device__ __forceinline__ float mac(const float4 &a, const float4 &w, float v) {
    return fmaf(a.w, w.w, fmaf(a.z, w.z, fmaf(a.y, w.y, fmaf(a.x, w.x, v))));
}
__device__ __forceinline__ double mac(const double2 &a, const double2 &w, double v) {
    return fma(a.y, w.y, fma(a.x, w.x, v));
}
template <typename T> struct Vec;                 // 16 bytes of K
template <> struct Vec<float> { using type = float4; };
template <> struct Vec<double> { using type = double2; };

// 16-byte copy, zero-filled without a source
__device__ __forceinline__ void copy16(uint32_t dst, const void *src, bool have) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(have ? 16 : 0) : "memory");
}

// A tile of the level's row list may be taller than BM (the tensor-core tiles are 128 rows):
// blockIdx.x enumerates (tile, BM-row slice) pairs, `subs` slices per tile.
template <typename T>
__global__ void __launch_bounds__(THREADS) gemm_simt_kernel(const __grid_constant__ GemmDev g, int subs) {
    constexpr int BK = 64 / (int)sizeof(T);       // values of K per stage
    constexpr int BN = kCols<T>, NJ = BN / 8, kStageBytes = (BM + BN) * kPitch;
    using V = typename Vec<T>::type;
    __shared__ __align__(16) unsigned char sm[kStages * kStageBytes];
    const Tile t = g.tiles[blockIdx.x / subs];
    const int r_off = (blockIdx.x % subs) * BM;     // first tile row of this slice
    const int nrows = min(BM, t.nrows - r_off);     // may be <= 0 for a short tile
    if (nrows <= 0) return;
    const int n0 = blockIdx.y * BN, tid = threadIdx.x;
    const int tr = tid >> 3, tc = tid & 7;          // its rows tr + 16 i, columns tc + 8 j
    const int nseg = gemm_nseg(g);
    // copies: unit q of rows lrow and lrow + 32, of A and of W
    const int lrow = tid >> 2, q = tid & 3;
    const int box0 = lrow < nrows ? gemm_row_box(g, t, r_off + lrow) : -1;
    const int box1 = lrow + 32 < nrows ? gemm_row_box(g, t, r_off + lrow + 32) : -1;
    const uint32_t sd = smem_u32(sm) + lrow * kPitch + q * 16;
    const bool wok0 = n0 + lrow < g.n_out, wok1 = n0 + lrow + 32 < g.n_out;
    // the copy position: segment, its sources, first value of K
    int seg = -1, k = 0, K = 0, s0 = -1, s1 = -1;
    const T *X = nullptr, *W = nullptr;
    int ldx = 0;
    auto next_segment = [&]() {                     // to the next segment with any product; false at the end
        for (++seg; seg < nseg; ++seg)
            if (gemm_seg_active(g, t, seg) && gemm_seg_k(g, seg) > 0) break;
        if (seg >= nseg) return false;
        const bool second = g.mode == GM_PARENT2 && seg == 1;
        X = (const T *)(second ? g.X1 : g.X0);
        ldx = second ? g.ldx1 : g.ldx0;
        K = gemm_seg_k(g, seg);
        W = second ? (const T *)g.W1[t.cls] : (const T *)g.W0 + gemm_w_index(g, t, seg) * g.w_stride;
        s0 = box0 >= 0 ? gemm_src_row(g, t, box0, seg) : -1;
        s1 = box1 >= 0 ? gemm_src_row(g, t, box1, seg) : -1;
        k = 0;
        return true;
    };
    bool more = next_segment();
    auto copy_stage = [&](int stage) {              // one chunk, or an empty group at the end
        if (more) {
            const uint32_t d = sd + stage * kStageBytes;
            const int kq = k + q * (16 / (int)sizeof(T));   // K is a multiple of 16: whole chunks
            copy16(d, X + (size_t)max(s0, 0) * ldx + kq, s0 >= 0);
            copy16(d + 32 * kPitch, X + (size_t)max(s1, 0) * ldx + kq, s1 >= 0);
            const T *w = W + (size_t)(n0 + lrow) * K + kq;
            copy16(d + BM * kPitch, wok0 ? w : W, wok0);
            if (BN > 32) copy16(d + (BM + 32) * kPitch, wok1 ? w + (size_t)32 * K : W, wok1);
            k += BK;
            if (k >= K) more = next_segment();
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // chunks in all
    int chunks = 0;
    for (int s = 0; s < nseg; ++s)
        if (gemm_seg_active(g, t, s)) chunks += (gemm_seg_k(g, s) + BK - 1) / BK;
    T acc[4][NJ];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0;
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) copy_stage(s);
    const unsigned char *pa = sm + tr * kPitch, *pw = sm + (BM + tc) * kPitch;
    int stage = 0;
    for (int c = 0; c < chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();
        copy_stage(stage == 0 ? kStages - 1 : stage - 1);   // the stage read in the last iteration
        const unsigned char *sa = pa + stage * kStageBytes, *sw = pw + stage * kStageBytes;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            V a[4], w[NJ];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const V *>(sa + 16 * i * kPitch + u * 16);
#pragma unroll
            for (int j = 0; j < NJ; ++j) w[j] = *reinterpret_cast<const V *>(sw + 8 * j * kPitch + u * 16);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = mac(a[i], w[j], acc[i][j]);
        }
        stage = stage + 1 == kStages ? 0 : stage + 1;
    }
    T *Y = (T *)g.Y;
    const T alpha = sizeof(T) == 8 ? (T)g.alpha_d : (T)g.alpha;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = tr + 16 * i;
        if (r >= nrows) continue;
        const int b = gemm_row_box(g, t, r_off + r);
        T *y = Y + (size_t)b * g.ldy + n0 + tc;
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            if (n0 + tc + 8 * j < g.n_out) {
                const T v = alpha * acc[i][j];
                y[8 * j] = g.accumulate ? y[8 * j] + v : v;
            }
    }
}

}  // namespace

GemmDev make_gemm_dev(const fmm_ctx *ctx, const GemmCall &c);

template <typename T>
cudaError_t gemm_simt(const fmm_ctx *ctx, const GemmCall &c, cudaStream_t s) {
    GemmDev g = make_gemm_dev(ctx, c);
    const TileSet &ts = c.tiles ? *c.tiles
                        : (c.mode == GM_STENCIL || c.mode == GM_PARENT2) ? ctx->tiles_cls[c.level]
                                                                         : ctx->tiles_plain[c.level];
    if (ts.ntiles == 0) return cudaSuccess;
    // whole chunks of K, rows of whole 16-byte units (every caller's are padded to 16 values)
    if ((c.k0 & 15) || (c.ldx0 & 3) || (c.X1 && ((c.k1 & 15) || (c.ldx1 & 3))) || ((uintptr_t)c.X0 & 15) ||
        ((uintptr_t)c.X1 & 15))
        return cudaErrorInvalidValue;
    g.tiles = ts.tiles;
    g.masks = ts.masks;
    if (c.mode == GM_STENCIL && ctx->masks_ev) {   // the masks are computed on a side stream
        cudaError_t e = cudaStreamWaitEvent(s, ctx->masks_ev, 0);
        if (e != cudaSuccess) return e;
    }
    const int tm = ts.tile_m ? ts.tile_m : ctx->tile_m;
    const int subs = (tm + BM - 1) / BM;
    dim3 grid(ts.ntiles * subs, (c.n_out + kCols<T> - 1) / kCols<T>);
    gemm_simt_kernel<T><<<grid, THREADS, 0, s>>>(g, subs); count_launch();
    return cudaGetLastError();
}

template cudaError_t gemm_simt<float>(const fmm_ctx *, const GemmCall &, cudaStream_t);
template cudaError_t gemm_simt<double>(const fmm_ctx *, const GemmCall &, cudaStream_t);

}  // namespace fmm
