// FP64 M2L stencil on the FP16 tensor cores (tcgen05, sm_103a), exact products from integer digits.
//
// FP64 arithmetic runs at 1.25 TFLOP/s on this part, the FP16 tensor pipe at 2,000, so the stencil's
// products are cut into integers that the tensor pipe multiplies and adds without rounding (the error-free
// splitting of a matrix product into slices of Ozaki, Ogita, Oishi and Rump, 2012).  A row is
// scaled by a power of two to at most 64 in size and written as eight digits of 7 bits, x = sum_i
// d_i 2^(-7 i) with integers |d_i| <= 64 (56 bits below the row's largest entry; FP16 holds every
// digit exactly), an operator likewise.  The products of digits i and j have the weight 2^(-7 (i + j));
// those of i + j <= 7 are kept (36 of 64; the others are below 2^-56 of the largest product).  All
// products of one weight, over all of K, add up in one tensor-memory accumulator: at most 8 K 2^12,
// below 2^24 for K <= 504, so that every FP32 sum is an exact integer.  A drain warp joins the eight
// sums of an output to two 52-bit integers and adds them, times their scales, to an FP64 sum: four
// FP64 operations for the 2 K of the direct form.  Precision: <A q, g> - <q, A^T g>, which is zero in
// exact arithmetic, is 4.3e-18 of |A q| |g| on 30,011 cube points (p = 6, depth 3; 1.2e-17 with FP64
// products) and smaller than with FP64 products on every case tried; potentials differ from those by
// 1.5e-15.
//
// Layout.  One CTA computes a 128-row tile (the boxes of one octant) for 64 output columns: eight
// accumulators of 64 columns fill the tensor memory.  blockIdx.y splits the columns, blockIdx.z cuts
// the 189 transfer vectors into groups whose partial sums go to memory.  A stage holds 16 values of
// K: eight A planes of 32-byte rows (SWIZZLE_32B) and eight operator planes without swizzle, 48 KB,
// four stages.  Rows lie in memory as [row][16 of K][digit][16 values], 256 contiguous bytes a stage.
//
// Warps (448 threads): 0-3 copy A rows, 4 issues, 5 loads operators, 6-13 drain (two a lane quarter,
// 32 columns each).  What bounds it: a transfer vector takes 36 MMAs of 48 cycles per 16 of K (15,600
// cycles at K = 144), then 16,400 cycles of FP64 additions before the accumulators are free again.
// M2L of 100,003 cube points, p = 6, depth 4: 41.4 ms with FP64 products -> 4.4 ms.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "gemm_common.cuh"
#include "tcgen05.cuh"

namespace fmm {

namespace {

constexpr int kDig = 8;                // digits, and weights kept
constexpr int kRows = 128, kCols = 64; // tile rows, output columns per CTA
constexpr int kChunk = 16;             // values of K per stage
constexpr int kStages = 4;
constexpr int kAPlane = kRows * kChunk * 2, kBPlane = kCols * kChunk * 2;
constexpr int kStageBytes = kDig * (kAPlane + kBPlane);
constexpr int kProducers = 128, kIssuer = 4, kLoader = 5, kDrain0 = 6, kThreads = 448;
constexpr int kHalf = kCols / 2;       // columns a drain thread holds
constexpr int kRing = 8;               // segments whose row exponents are kept (stages + 2 at least)
constexpr int kNone = -(1 << 30), kBad = 1 << 30;   // exponents: no source or a zero row; a row that is not finite

struct F64Dev {
    GemmDev g;
    const unsigned char *xp;    // digit rows: ld bytes a row
    long long ld;
    const int *xe;              // exponent per row
    const unsigned char *w;     // operators: [nsplit][K / 16][digit][2 units][64][16 B], w_op bytes each
    long long w_op;
    const int *we;              // exponent per operator
    int K;
    int groups;
    double *Y;
    int ldy;
    long long y_group;
    int *err;
    unsigned long long wait_ns;
};

struct Seg {
    short slot, delta;
    int op;
};

// the eight digits of y, |y| <= 64, as FP16 integers
__device__ __forceinline__ void digits(double y, __half *d) {
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
        const double r = rint(y);
        d[i] = __double2half(r);
        y = (y - r) * 128.0;
    }
}

__device__ __forceinline__ int exponent_of(double m) {   // m < 2^e
    int e = 0;
    frexp(m, &e);
    return e;
}

__global__ void __launch_bounds__(kThreads, 1) gemm_f64_kernel(const __grid_constant__ F64Dev p) {
    extern __shared__ unsigned char smem_raw[];
    // (as gemm_f16.cu's; ring: the row exponents of a slot written, one arrival a producer warp)
    __shared__ uint64_t full_bar[kStages], empty_bar[kStages], tfull_bar, tempty_bar, fin_bar, ring_bar[kRing];
    __shared__ uint32_t tmem_base;
    __shared__ int box[kRows];
    __shared__ int ring[kRing][kRows];
    __shared__ Seg seg[kClassSlots];
    __shared__ uint32_t mask[6];
    __shared__ int abort_flag, started_items;

    const GemmDev &g = p.g;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const Tile t = g.tiles[blockIdx.x];
    const int n_lo = blockIdx.y * kCols, nch = p.K / kChunk;
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full_bar[s], kProducers + 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&tfull_bar, 1), mbar_init(&tempty_bar, 8), mbar_init(&fin_bar, 1);
        for (int k = 0; k < kRing; ++k) mbar_init(&ring_bar[k], kProducers / 32);
        abort_flag = started_items = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int lo = kClassSlots * (int)blockIdx.z / p.groups, hi = kClassSlots * ((int)blockIdx.z + 1) / p.groups;
    if (tid < 6) {
        const int b0 = max(lo - 32 * tid, 0), b1 = min(hi - 32 * tid, 32);
        const uint32_t keep = b1 <= b0 ? 0u : (b1 == 32 ? 0xffffffffu : (1u << b1) - 1u) & ~((1u << b0) - 1u);
        mask[tid] = g.masks[(size_t)t.mask * 6 + tid] & keep;
    }
    if (tid < kRows) box[tid] = tid < t.nrows ? gemm_row_box(g, t, tid) : -1;
    __syncwarp();
    if (warp == 0) tmem_alloc(&tmem_base, 512);
    __syncthreads();
    int nact = 0;
#pragma unroll
    for (int w = 0; w < 6; ++w) nact += __popc(mask[w]);
    if (tid < kClassSlots && ((mask[tid >> 5] >> (tid & 31)) & 1u)) {
        int pos = __popc(mask[tid >> 5] & ((1u << (tid & 31)) - 1u));
        for (int w = 0; w < (tid >> 5); ++w) pos += __popc(mask[w]);
        seg[pos] = Seg{(short)tid, (short)g.class_delta[t.cls * kClassSlots + tid], g.class_slots[t.cls * kClassSlots + tid]};
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp < 4) {
        // ------------------------------------------------------------ producers
        // Lane l looks up its warp's row l; the warp copies four rows a pass: lane (digit, row, unit)
        // = (l / 8, l / 2 mod 4, l mod 2), and the digit's partner four above.
        const int dig = lane >> 3, r4 = (lane >> 1) & 3, u = lane & 1;
        const int row = tid;
        int ax = 0, ay = 0, az = 0;
        const int mybox = box[row];
        if (mybox >= 0) demorton3(g.keys[mybox], ax, ay, az);
        auto source = [&](int i) {
            if (mybox < 0) return -1;
            int dx, dy, dz;
            unpack_delta(seg[i].delta, dx, dy, dz);
            return dense_find(g.dense, g.level, ax + dx, ay + dy, az + dz);
        };
        const uint32_t sd = smem_u32(base) + dig * kAPlane + (warp * 32 + r4) * 32 + u * 16;
        int arrived = 0, stage = 0, slot = 0;
        uint32_t phase = 1;
        bool ok = true;
        int src = nact > 0 ? source(0) : -1;
        for (int i = 0; i < nact; ++i) {
            const int next = i + 1 < nact ? source(i + 1) : -1;
            const int xe = src >= 0 ? __ldg(p.xe + src) : kNone, we = __ldg(p.we + seg[i].op);
            ring[slot][row] = xe == kNone || we == kNone ? kNone : xe == kBad || we == kBad ? kBad : xe + we;
            __syncwarp();
            if (lane == 0) mbar_arrive(&ring_bar[slot]);
            slot = (slot + 1) % kRing;
            int from[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) from[k] = __shfl_sync(0xffffffffu, src, 4 * k + r4);
            ok = __all_sync(0xffffffffu, ok && !*(volatile int *)&abort_flag);
            for (int c = 0; c < nch && ok; ++c) {
                if (!mbar_wait_warp(&empty_bar[stage], phase, p.wait_ns)) {
                    ok = false;
                    break;
                }
                const unsigned char *x = p.xp + (size_t)c * (kDig * 32) + dig * 32 + u * 16;
                const uint32_t d = sd + stage * kStageBytes;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (from[k] >= 0) {
                        const unsigned char *a = x + (size_t)from[k] * p.ld;
                        // rows 4 k + r4 of the warp: the swizzle exchanges the units of every other four rows
                        const uint32_t dd = (d ^ (k & 1 ? 16u : 0u)) + 128 * k;
                        cp_async16(dd, a);
                        cp_async16(dd + 4 * kAPlane, a + 128);
                    }
                cp_async_arrive(&full_bar[stage]);
                ++arrived;
                if (++stage == kStages) stage = 0, phase ^= 1u;
            }
            src = next;
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        // nothing may still be in flight when the CTA exits (as in gemm_f16.cu)
        cp_async_wait_all();
        __syncwarp();
        asm volatile("bar.sync 1, 160;" ::: "memory");
        const int started = started_items;
        for (int k = arrived; k < started; ++k) mbar_arrive(&full_bar[k % kStages]);
    } else if (warp == kLoader) {
        // ------------------------------------------------------------ operator copies
        int started = 0;
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 1;
            bool ok = true;
            for (int i = 0; i < nact && ok; ++i) {
                const unsigned char *w = p.w + (size_t)seg[i].op * p.w_op + (size_t)blockIdx.y * nch * kDig * kBPlane;
                for (int c = 0; c < nch; ++c) {
                    if (!mbar_wait(&empty_bar[stage], phase, p.wait_ns) || *(volatile int *)&abort_flag) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_tx(&full_bar[stage], kDig * kBPlane);
                    bulk_g2s(base + (size_t)stage * kStageBytes + kDig * kAPlane, w + (size_t)c * kDig * kBPlane,
                             kDig * kBPlane, &full_bar[stage]);
                    ++started;
                    if (++stage == kStages) stage = 0, phase ^= 1u;
                }
            }
            if (!ok) {
                atomicExch(p.err, FMM_ETIMEOUT);
                *(volatile int *)&abort_flag = 1;
            }
            started_items = started;
        }
        __syncwarp();
        asm volatile("bar.sync 1, 160;" ::: "memory");
        if (lane == 0)
            for (int k = max(0, started - kStages); k < started; ++k)
                if (!mbar_wait(&full_bar[k % kStages], (k / kStages) & 1, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
        __syncwarp();
    } else if (warp == kIssuer) {
        // ------------------------------------------------------------ MMA issuer
        const uint32_t elected = elect_one(), idesc = make_idesc(kCols, 0);
        const int n = __shfl_sync(0xffffffffu, nact, 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), sbase = smem_u32(base);
        bool ok = true;
        int stage = 0;
        uint32_t phase = 0, aphase = 1;
        for (int i = 0; i < n && ok; ++i) {
            for (int c = 0; c < nch; ++c) {
                const bool ready = mbar_wait(&full_bar[stage], phase, p.wait_ns) &&
                                   (c > 0 || mbar_wait(&tempty_bar, aphase, p.wait_ns)) && !*(volatile int *)&abort_flag;
                if (!__all_sync(0xffffffffu, ready)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                fence_proxy_async();
                const uint32_t sa = sbase + (uint32_t)(stage * kStageBytes), sb = sa + kDig * kAPlane;
                const uint64_t ad = sw32_desc(sa), bd = plain_desc(sb, kCols * 16);
#pragma unroll
                for (int w = 0; w < kDig; ++w)
#pragma unroll
                    for (int a = 0; a <= w; ++a)
                        mma_f16_elected(tm + (uint32_t)(w * kCols), ad + (uint64_t)(a * (kAPlane >> 4)),
                                        bd + (uint64_t)((w - a) * (kBPlane >> 4)), idesc, c > 0 || a > 0 ? 1u : 0u, elected);
                if (elected) {
                    mma_commit(&empty_bar[stage]);
                    if (c + 1 == nch) mma_commit(&tfull_bar);
                }
                __syncwarp();
                if (++stage == kStages) stage = 0, phase ^= 1u;
            }
            aphase ^= 1u;
        }
        if (elected) {
            if (!ok) {
                atomicExch(p.err, FMM_ETIMEOUT);
                *(volatile int *)&abort_flag = 1;
            }
            mma_commit(&fin_bar);
            if (!mbar_wait(&fin_bar, 0, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ drain and epilogue
        const int q = warp & 3, hf = (warp - kDrain0) >> 2, c0 = hf * kHalf;
        const int row = q * 32 + lane;
        double acc[kHalf];
#pragma unroll
        for (int i = 0; i < kHalf; ++i) acc[i] = 0.0;
        bool ok = true;
        int slot = 0;
        uint32_t phase = 0, rphase = 0;
        for (int i = 0; i < nact && ok; ++i) {
            if (!mbar_wait_warp(&tfull_bar, phase, p.wait_ns) || !mbar_wait_warp(&ring_bar[slot], rphase, p.wait_ns)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const int e = ring[slot][row];
            const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {   // weights 0-3, then 4-7
                // 2^(e - 12): both scales leave entries of at most 64 = 2^6
                const double f = e == kBad ? __longlong_as_double(0x7ff8000000000000ll)
                                           : e == kNone ? 0.0 : scalbn(1.0, e - 12 - (h ? 49 : 21));
#pragma unroll
                for (int n = 0; n < kHalf; n += 8) {
                    uint32_t v[4][8];
#pragma unroll
                    for (int k = 0; k < 4; ++k) tmem_ld8(ta + (uint32_t)((4 * h + k) * kCols + n), v[k]);
                    tmem_wait_ld();
                    if (e != kNone) {
#pragma unroll
                        for (int x = 0; x < 8; ++x) {
                            // exact integers below 2^24, weights 2^21, 2^14, 2^7 and 1
                            const int i0 = __float2int_rn(__uint_as_float(v[0][x])), i1 = __float2int_rn(__uint_as_float(v[1][x]));
                            const int i2 = __float2int_rn(__uint_as_float(v[2][x])), i3 = __float2int_rn(__uint_as_float(v[3][x]));
                            const long long s = (long long)(i0 * 128 + i1) * 16384 + (i2 * 128 + i3);
                            // |s| < 2^51: its bits added to 3 * 2^51 read as a double, less 3 * 2^51
                            const double d = __longlong_as_double(0x4338000000000000ll + s) - 6755399441055744.0;
                            acc[n + x] = fma(f, d, acc[n + x]);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty_bar);
            phase ^= 1u;
            if (++slot == kRing) slot = 0, rphase ^= 1u;
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        const int b = row < t.nrows ? box[row] : -1;
        if (ok && b >= 0) {
            double *y = p.Y + (size_t)blockIdx.z * p.y_group + (size_t)b * p.ldy + n_lo + c0;
#pragma unroll
            for (int n = 0; n < kHalf; n += 2)
                if (n_lo + c0 + n < g.n_out) *reinterpret_cast<double2 *>(y + n) = make_double2(acc[n], acc[n + 1]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Rows list[i] (i without a list) of FP64 values to digits and an exponent.  One warp per row; lane l
// takes the 16 values of chunks l, l + 32, ..
__global__ void __launch_bounds__(256)
digit_rows_kernel(const double *__restrict__ x, int ldx, const int *__restrict__ list, int nrows, int K,
                  unsigned char *__restrict__ out, long long ld, int *__restrict__ exps) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= nrows) return;
    const int r = list ? list[i] : i;
    const double *xr = x + (size_t)r * ldx;
    double m = 0;
    int bad = 0;
    for (int k = lane; k < K; k += 32) {
        const double v = fabs(xr[k]);
        bad |= !(v <= 1.7976931348623157e308);
        m = fmax(m, v);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    bad = __any_sync(0xffffffffu, bad);
    const int e = bad ? kBad : m > 0 ? exponent_of(m) : kNone;
    if (lane == 0) exps[r] = e;
    unsigned char *o = out + (size_t)r * ld;
    for (int k = lane; k < K; k += 32) {
        const double v = xr[k];
        __half d[kDig];
        digits(bad || m == 0 ? 0.0 : scalbn(v, 6 - e), d);
#pragma unroll
        for (int g = 0; g < kDig; ++g)
            *reinterpret_cast<__half *>(o + (size_t)(k >> 4) * (kDig * 32) + g * 32 + (k & 15) * 2) = d[g];
    }
}

// Operator k (block k): rows x cols FP64 to digits in the stage form and its exponent.
__global__ void __launch_bounds__(256)
digit_pack_kernel(const double *__restrict__ w, int rows, int cols, int nsplit, int K, unsigned char *__restrict__ out,
                  int *__restrict__ exps) {
    __shared__ double red[256];
    const double *a = w + (size_t)blockIdx.x * rows * cols;
    double m = 0;
    for (int i = threadIdx.x; i < rows * cols; i += 256) m = fmax(m, fabs(a[i]));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    const int e = red[0] > 0 ? exponent_of(red[0]) : kNone;
    if (threadIdx.x == 0) exps[blockIdx.x] = e;
    const int nch = K / kChunk, total = nsplit * kCols * K;
    unsigned char *o = out + (size_t)blockIdx.x * total * 2 * kDig;
    for (int i = threadIdx.x; i < total; i += 256) {
        const int n = i / K, k = i % K, ns = n / kCols, r = n % kCols, c = k / kChunk, kin = k % kChunk;
        const double v = n < rows && k < cols && e != kNone ? scalbn(a[(size_t)n * cols + k], 6 - e) : 0.0;
        __half d[kDig];
        digits(v, d);
        unsigned char *at = o + ((size_t)ns * nch + c) * (kDig * kBPlane) + ((kin >> 3) * kCols + r) * 16 + (kin & 7) * 2;
#pragma unroll
        for (int g = 0; g < kDig; ++g) *reinterpret_cast<__half *>(at + g * kBPlane) = d[g];
    }
}

// y[r] = sum of the groups' partial rows in order, rows list[i] (i without a list); one thread per two values
__global__ void group_sum_kernel(const double *__restrict__ x, long long x_group, int groups, int ld,
                                 const int *__restrict__ list, int nrows, int ncols, double *__restrict__ y, int ldy) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int per = ncols / 2;
    if (i >= (long long)nrows * per) return;
    const int q = (int)(i / per), c = 2 * (int)(i % per), r = list ? list[q] : q;
    double2 s = *reinterpret_cast<const double2 *>(x + (size_t)r * ld + c);
    for (int k = 1; k < groups; ++k) {
        const double2 a = *reinterpret_cast<const double2 *>(x + k * x_group + (size_t)r * ld + c);
        s.x += a.x, s.y += a.y;
    }
    *reinterpret_cast<double2 *>(y + (size_t)r * ldy + c) = s;
}

}  // namespace

bool f64_stencil_ok(int K) { return K <= 504; }   // 8 K 2^12 < 2^24: every sum of digit products is exact

cudaError_t f64_upload(fmm_ctx *ctx, const double *w, int count, int rows, int cols, int K, F64Mat *out) {
    out->K = K, out->nsplit = (round_up(rows, 16) + kCols - 1) / kCols;
    out->op_bytes = (size_t)out->nsplit * kCols * K * 2 * kDig;
    void *d = nullptr, *e = nullptr;
    FMM_CUDA_TRY(dev_malloc(&d, out->op_bytes * count));
    ctx->op_allocs.push_back(d);
    FMM_CUDA_TRY(dev_malloc(&e, count * sizeof(int)));
    ctx->op_allocs.push_back(e);
    cudaStream_t s = ctx->stream;
    Scratch<double> tmp;
    FMM_CUDA_TRY(tmp.alloc((size_t)count * rows * cols, s));
    FMM_CUDA_TRY(cudaMemcpyAsync(tmp.p, w, (size_t)count * rows * cols * sizeof(double), cudaMemcpyHostToDevice, s));
    digit_pack_kernel<<<count, 256, 0, s>>>(tmp.p, rows, cols, out->nsplit, K, (unsigned char *)d, (int *)e);
    count_launch();
    FMM_CUDA_TRY(cudaGetLastError());
    FMM_CUDA_TRY(cudaStreamSynchronize(s));   // the host operators may be released
    out->data = d, out->exps = (int *)e;
    return cudaSuccess;
}

GemmDev make_gemm_dev(const fmm_ctx *ctx, const GemmCall &c);

cudaError_t stencil_f64(const fmm_ctx *ctx, const GemmCall &c, const F64Mat &W, const int *source_list, int64_t n_source,
                        unsigned char *digit_rows, int *exps, const int *list, int64_t n_rows, double *partial,
                        cudaStream_t s) {
    const TileSet &ts = c.tiles ? *c.tiles : ctx->tiles_cls[c.level];
    if (ts.ntiles == 0) return cudaSuccess;
    const long long ld = (long long)W.K * 2 * kDig;
    if (W.K > c.ldx0 || (c.ldy & 1) || ((uintptr_t)digit_rows & 15) || ((uintptr_t)c.Y & 15)) return cudaErrorInvalidValue;
    if (n_source > 0) {
        digit_rows_kernel<<<(unsigned)((n_source + 7) / 8), 256, 0, s>>>((const double *)c.X0, c.ldx0, source_list, (int)n_source,
                                                                         W.K, digit_rows, ld, exps);
        count_launch();
        FMM_CUDA_TRY(cudaGetLastError());
    }
    F64Dev p{};
    p.g = make_gemm_dev(ctx, c);
    p.g.tiles = ts.tiles;
    p.g.masks = ts.masks;
    if (ctx->masks_ev) FMM_CUDA_TRY(cudaStreamWaitEvent(s, ctx->masks_ev, 0));
    p.xp = digit_rows, p.ld = ld, p.xe = exps;
    p.w = (const unsigned char *)W.data, p.w_op = (long long)W.op_bytes, p.we = W.exps;
    p.K = W.K;
    p.groups = c.groups;
    p.Y = c.groups > 1 ? partial : (double *)c.Y;
    p.ldy = c.ldy, p.y_group = c.y_group;
    p.err = ctx->dev_flag, p.wait_ns = ctx->tc_wait_ns;
    const size_t smem = (size_t)kStages * kStageBytes + 1024;
    FMM_CUDA_TRY(allow_all_shared(gemm_f64_kernel));
    gemm_f64_kernel<<<dim3(ts.ntiles, W.nsplit, c.groups), kThreads, smem, s>>>(p);
    count_launch();
    FMM_CUDA_TRY(cudaGetLastError());
    if (c.groups == 1) return cudaSuccess;
    const long long n2 = (long long)n_rows * (c.n_out / 2);
    if (n2 == 0) return cudaSuccess;
    group_sum_kernel<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(partial, c.y_group, c.groups, c.ldy, list, (int)n_rows,
                                                                   c.n_out, (double *)c.Y, c.ldy);
    count_launch();
    return cudaGetLastError();
}

}  // namespace fmm
