// Gathered GEMM of gemm_common.cuh on the tensor cores (tcgen05, sm_103a) from FP16 planes.
//
// Operands.  Rows and operators are scaled by powers of two (largest entry just below 2^14) and cut
// into FP16 terms of 11 bits each: two planes (hi, lo: 22 bits; FMM_FP16X3, products lo*hi, hi*lo,
// hi*hi) or three (hi, mid, lo: 33 bits, which holds an FP32 value exactly unless it is more than 2^14
// below the row's largest; FMM_FP32's M2L in shallow and in adaptive trees, the six products of order
// below three).  Rows and operators of two planes have a scale per 64 columns; those of three planes, and
// the stencil's where the compressed vectors fit one CTA, one for the whole row or operator.  The products
// add up in FP32 in tensor memory, smallest products first; since the tensor core truncates when it adds,
// an accumulator takes one chunk's MMAs (at most four of them the large products) before it is multiplied
// by its scales and added, correctly rounded, into FP32 registers.  Where the stencil of two planes has one
// scale a row, all chunks of a transfer vector add up in one accumulator.
//
// Layout.  One CTA computes a 128-row tile for ncta <= 160 output columns; blockIdx.y splits wider
// outputs, blockIdx.z cuts the 189 transfer vectors of a stencil into groups whose partial sums go
// to memory (stencil_groups).  K is cut into chunks of at most 64 (two planes) or 32 (three); three to
// six stages fill the 227 KB of shared memory, since a stage's copies take about 1 us from L2 and its
// MMAs 0.4 us.  A stage holds the A planes as K-major rows of 128 B (SWIZZLE_128B) or 64 B
// (SWIZZLE_64B), so that the 16-byte copies of a row write one line (unswizzled, with the units of a
// row 2 KB apart, the same copies took 1.6 us a chunk instead of 0.8), and the operator without swizzle,
// [plane][16-byte unit of K][column][16 B] (LBO = columns * 16 B, SBO = 128 B), as it lies in global
// memory: one bulk copy a chunk.
//
// Warps (480 threads, one CTA an SM): 0-3 copy A rows by cp.async, 4 and 5 issue the MMAs in turn,
// 6-13 drain, two a lane quarter, each half of the columns, 14 loads operators.
//
// What bounds it: the tensor pipe on full tiles (eval on 4.2M cube points, p = 8: 0.6 us a chunk of 960
// MMA cycles), the producers' instructions where most rows are absent (the sphere: 0.5 us a chunk of
// 720; there the tensor pipe is busy 54% of the time).  M2L of all levels, far field alone, against the
// kernel with two 72 KB stages and products issued by one lane: sphere 8.39M p = 6 3.25 -> 1.63 ms, cube
// 1M p = 6 1.89 -> 0.75 ms, cube 4.2M p = 8 53.6 -> 14.9 ms.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "gemm_common.cuh"
#include "tcgen05.cuh"

namespace fmm {

namespace {

constexpr int kRows = 128;
constexpr int kMaxCols = 160;          // output columns per CTA
constexpr int kProdWarps = 4, kProducers = 32 * kProdWarps, kWarpRows = 32;   // warps 0-3, a row a thread
static_assert(kProdWarps * kWarpRows == kRows);
constexpr int kIssuer = 4;             // warps 4 and 5
constexpr int kDrain0 = 6;             // warps 6-13
constexpr int kLoader = 14;
constexpr int kThreads = 480;
constexpr int kHalf = kMaxCols / 2;    // columns a drain thread holds at most
constexpr int kMaxStages = 6;
constexpr int kMaxChunks = 32;         // of one operator (K <= 992 in chunks of 32 or more)
constexpr int kAcc = 3;                // tensor-memory accumulators
// Segments (or chunks) whose row factors are kept: the producers run at most (stages + accumulators +
// 2) chunks ahead of the slowest drain warp.
constexpr int kFacRing = kMaxStages + kAcc + 3;

// A planes in shared memory: K-major rows of 128 B (64 values, SWIZZLE_128B) with two planes, of 64 B
// (32 values, SWIZZLE_64B) with three.  16-byte unit u of row r lies at a_offset(r, u).
template <int NPL> constexpr int kRowBytes = NPL == 2 ? 128 : 64;
template <int NPL> __device__ __forceinline__ uint32_t a_offset(int r, int u) {
    return NPL == 2 ? r * 128 + ((u ^ (r & 7)) << 4) : r * 64 + ((u ^ ((r >> 1) & 3)) << 4);
}

// One operand pair: A rows from planes, operators packed by f16_upload.
struct F16Seg {
    const unsigned char *xp;    // planes of the A rows
    long long xplane;           // bytes between planes
    int ld;                     // row stride in elements
    const float *xs;            // 1 / scale per row, or per row and chunk: nxs values a row
    int nxs;
    const unsigned char *w;     // operators
    long long w_op;             // bytes per operator
    const float *ws;            // 1 / scale per operator (and chunk, as the rows)
    int K, chunk, nch;
};

struct F16Dev {
    GemmDev g;
    F16Seg s0, s1;              // s1: the parent rows of PARENT2
    int ncta;                   // columns per CTA (operators padded to nsplit * ncta rows)
    int nstages, stage_bytes;
    int tmem_cols;
    int groups;                 // gridDim.z: groups of transfer vectors
    // Both segments' rows and operators are scaled per chunk.  (Whether one is says nothing of the other: a
    // segment of one chunk has one scale a row in either form.)
    int chunked;
    int seg_acc;                // a segment's chunks add up in one accumulator (one scale a row and operator)
    float *Y;                   // FP32 rows (of group z: Y + z * y_group), or null
    int ldy;
    long long y_group;
    unsigned char *yp;          // FP16 planes of the rows (nsplit == 1, groups == 1), or null
    long long yplane;
    int ldyp;
    float *ys;                  // 1 / scale of every row of yp, or per row and 64 columns: nys values a row
    int nys;
    int *err;
    unsigned long long wait_ns;
};

// 1 / scale and scale (powers of two) of a row whose largest |entry| has the bits m: the scaled
// entries are below 2^14.  A row of zeros has 1 / scale 0 (its products are skipped); a row with
// an infinity or NaN keeps scale 1, so that its planes and every result they enter are not finite.
__device__ __forceinline__ void row_scale(uint32_t m, float &scale, float &inv) {
    scale = inv = 1.f;
    if (m == 0u) inv = 0.f;
    else if (m < 0x7f800000u) {
        const int ex = max((int)(m >> 23), 1) - 126;            // the value is below 2^ex
        const int e = min(max(14 - ex, -126), 126);
        scale = __int_as_float((e + 127) << 23);
        inv = __int_as_float((127 - e) << 23);
    }
}

template <int NPL>
__device__ __forceinline__ void split_f16(float x, uint32_t *h) {
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
        const __half v = __float2half_rn(x);
        h[k] = __half_as_ushort(v);
        x -= __half2float(v);
    }
}

// Per-tile list of the active segments, in order.
struct SegTable {
    float ws[kClassSlots];       // 1 / scale of the segment's operator (one scale a row)
    short op[kClassSlots];
    short delta[kClassSlots];
    unsigned char seg[kClassSlots];
};

// One tile row: its box, its coordinates and, for neighbour keys, its Morton key's bits of each axis
// with the other axes' bits set, so that an addition carries from one bit of the axis to the next.
struct RowPos {
    int box, ax, ay, az;
    uint32_t sx, sy, sz;
};

constexpr uint32_t kAxis = 0x09249249u;   // every third bit, ten of them
// -3..3 spread to every third bit (two's complement of ten bits)
__constant__ uint32_t kSpreadDelta[7] = {0x09249241u, 0x09249248u, 0x09249249u, 0u, 1u, 8u, 9u};

__device__ __forceinline__ RowPos row_pos(const GemmDev &g, int box) {
    RowPos r{box, 0, 0, 0, 0u, 0u, 0u};
    if (box >= 0 && g.mode == GM_STENCIL) {
        const uint32_t k = g.keys[box];
        demorton3(k, r.ax, r.ay, r.az);
        r.sx = ((k >> 2) & kAxis) | ~kAxis, r.sy = ((k >> 1) & kAxis) | ~kAxis, r.sz = (k & kAxis) | ~kAxis;
    }
    return r;
}

// source row of (tile row, active segment i), -1 for none
__device__ __forceinline__ int source_row(const GemmDev &g, const SegTable &st, const RowPos &r, int i) {
    if (r.box < 0) return -1;
    switch (g.mode) {
        case GM_STENCIL: {
            const int d = st.delta[i], ix = d & 15, iy = (d >> 4) & 15, iz = (d >> 8) & 15;   // component + 3
            const uint32_t m = 1u << g.level;
            if ((uint32_t)(r.ax + ix - 3) >= m || (uint32_t)(r.ay + iy - 3) >= m || (uint32_t)(r.az + iz - 3) >= m)
                return -1;
            const uint32_t key = (((r.sx + kSpreadDelta[ix]) & kAxis) << 2) | (((r.sy + kSpreadDelta[iy]) & kAxis) << 1) |
                                 ((r.sz + kSpreadDelta[iz]) & kAxis);
            return g.dense[key];
        }
        case GM_CHILDREN: return g.child[(size_t)r.box * 8 + st.seg[i]];
        case GM_PARENT2: return st.seg[i] == 0 ? r.box : g.parent[r.box];
        default: return r.box;
    }
}

template <int NPL>
__global__ void __launch_bounds__(kThreads, 1) gemm_f16_kernel(const __grid_constant__ F16Dev p) {
    extern __shared__ unsigned char smem_raw[];
    // full: a stage's A copies (one arrival a producer thread) and its operator copy (the loader's
    // expect_tx arrival); empty: the stage's MMAs done; tfull / tempty: an accumulator's MMAs done
    // / drained; turn: an issuer may wait for its next chunk; fin: every MMA of an issuer done; fac: the
    // row factors of a slot written (one arrival a producer warp; the full barriers' arrivals follow the
    // asynchronous copies alone and make no ordinary store visible)
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tfull_bar[kAcc], tempty_bar[kAcc], turn_bar[2], fin_bar[2];
    __shared__ uint64_t fac_bar[kFacRing];
    __shared__ uint32_t tmem_base;
    __shared__ int box[kRows];
    __shared__ float fac[kFacRing][kRows];
    __shared__ SegTable st;
    __shared__ uint32_t mask[6];
    __shared__ int abort_flag, started_items;

    const GemmDev &g = p.g;
    // the warp's number in a form that the compiler knows to be the same in all lanes
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const Tile t = g.tiles[blockIdx.x];
    const int ncta = p.ncta, n_lo = blockIdx.y * ncta;
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

    if (tid == 0) {
        for (int s = 0; s < p.nstages; ++s) {
            mbar_init(&full_bar[s], kProducers + 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < kAcc; ++b) {
            mbar_init(&tfull_bar[b], 1);
            mbar_init(&tempty_bar[b], 8);
        }
        for (int k = 0; k < 2; ++k) mbar_init(&turn_bar[k], 1), mbar_init(&fin_bar[k], 1);
        for (int k = 0; k < kFacRing; ++k) mbar_init(&fac_bar[k], kProdWarps);
        abort_flag = 0;
        started_items = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // this group's segments: [lo, hi) of the mode's, the inactive slots of a stencil left out
    const int nseg_all = gemm_nseg(g);
    const int lo = (int)((long long)nseg_all * blockIdx.z / p.groups);
    const int hi = (int)((long long)nseg_all * (blockIdx.z + 1) / p.groups);
    if (tid < 6) {
        uint32_t m = g.mode == GM_STENCIL ? g.masks[(size_t)t.mask * 6 + tid] : 0xffffffffu;
        const int b0 = max(lo - 32 * tid, 0), b1 = min(hi - 32 * tid, 32);
        const uint32_t keep = b1 <= b0 ? 0u : (b1 == 32 ? 0xffffffffu : (1u << b1) - 1u) & ~((1u << b0) - 1u);
        mask[tid] = m & keep;
    }
    if (tid < kRows) box[tid] = tid < t.nrows ? gemm_row_box(g, t, tid) : -1;
    __syncwarp();
    if (warp == 0) tmem_alloc(&tmem_base, p.tmem_cols);
    __syncthreads();
    int nact = 0;
#pragma unroll
    for (int w = 0; w < 6; ++w) nact += __popc(mask[w]);
    if (tid < kClassSlots && ((mask[tid >> 5] >> (tid & 31)) & 1u)) {
        int pos = __popc(mask[tid >> 5] & ((1u << (tid & 31)) - 1u));
        for (int w = 0; w < (tid >> 5); ++w) pos += __popc(mask[w]);
        st.seg[pos] = (unsigned char)tid;
        int op = g.mode == GM_CHILDREN ? tid : 0;
        if (g.mode == GM_STENCIL) {
            op = g.class_slots[t.cls * kClassSlots + tid];
            st.delta[pos] = (short)g.class_delta[t.cls * kClassSlots + tid];
        }
        const bool second = g.mode == GM_PARENT2 && tid == 1;
        if (second) op = t.cls;
        st.op[pos] = (short)op;
        if (!p.chunked) st.ws[pos] = second ? p.s1.ws[op] : p.s0.ws[op];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    constexpr int aplane = kRows * kRowBytes<NPL>;   // bytes of an A plane in a stage
    auto seg_of = [&](int i) -> const F16Seg & { return g.mode == GM_PARENT2 && st.seg[i] == 1 ? p.s1 : p.s0; };

    if (warp < kProdWarps) {
        // ------------------------------------------------------------ producers
        // Lane l looks up the source of its warp's row l, a segment ahead of the copies; the warp then
        // copies its 32 rows, LPR lanes a row.
        constexpr int LPR = NPL == 2 ? 8 : 4, RPI = 32 / LPR, NP = kWarpRows / RPI;   // lanes a row, rows a pass, passes
        const int lr = lane / LPR, u = lane % LPR;               // its row of a pass and its unit
        const int row = warp * kWarpRows + lane;
        const uint32_t sd = smem_u32(base) + a_offset<NPL>(warp * kWarpRows + lr, u);
        const RowPos me = row_pos(g, box[row]);
        int arrived = 0, stage = 0;
        uint32_t phase = 1;        // of the stage's empty barrier (fresh: the phase before counts as done)
        bool ok = true;
        // src / xs: the row's source and its 1 / scale in this segment; src1: the source in the next.
        // Each is loaded a segment before it is used.
        int src = nact > 0 ? source_row(g, st, me, 0) : -1, src1 = nact > 1 ? source_row(g, st, me, 1) : -1;
        float xs = src >= 0 ? __ldg(seg_of(0).xs + (size_t)src * seg_of(0).nxs) : 0.f;
        const bool chunked = p.chunked;   // a factor per chunk instead of per segment
        int slot = 0;
        auto put_factor = [&](float f) {
            fac[slot][row] = f;
            __syncwarp();
            if (lane == 0) mbar_arrive(&fac_bar[slot]);
            slot = slot + 1 == kFacRing ? 0 : slot + 1;
        };
        for (int i = 0; i < nact; ++i) {
            const F16Seg &S = seg_of(i);
            if (!chunked) put_factor(xs * st.ws[i]);
            const int src2 = i + 2 < nact ? source_row(g, st, me, i + 2) : -1;
            const float xs1 = src1 >= 0 ? __ldg(seg_of(i + 1).xs + (size_t)src1 * seg_of(i + 1).nxs) : 0.f;
            int off[NP];   // in 16-byte units from the first row; negative: no source
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int r = __shfl_sync(0xffffffffu, src, k * RPI + lr);
                off[k] = r >= 0 ? r * (S.ld >> 3) + u : -1;
            }
            ok = __all_sync(0xffffffffu, ok && !*(volatile int *)&abort_flag);
            for (int c = 0; c < S.nch && ok; ++c) {
                if (chunked) {   // this chunk's factors; the next chunk's are loaded now
                    put_factor(xs);
                    if (c + 1 < S.nch) xs = src >= 0 ? __ldg(S.xs + (size_t)src * S.nxs + c + 1) : 0.f;
                }
                if (!mbar_wait_warp(&empty_bar[stage], phase, p.wait_ns)) {
                    ok = false;
                    break;
                }
                const int kv = min(S.chunk, S.K - c * S.chunk), units = kv >> 3;
                if (u < units) {
                    const unsigned char *x = S.xp + (size_t)c * S.chunk * 2;
                    const uint32_t d = sd + (uint32_t)(stage * p.stage_bytes);
#pragma unroll
                    for (int k = 0; k < NP; ++k)
                        if (off[k] >= 0) {
                            const unsigned char *a = x + (size_t)off[k] * 16;
#pragma unroll
                            for (int pl = 0; pl < NPL; ++pl)
                                // (rows 4 apart: the swizzle flips unit bit 2)
                                cp_async16((d ^ (NPL == 2 && (k & 1) ? 64u : 0u)) + (uint32_t)(k * RPI * kRowBytes<NPL> + pl * aplane),
                                           a + pl * S.xplane);
                        }
                }
                cp_async_arrive(&full_bar[stage]);
                ++arrived;
                if (++stage == p.nstages) stage = 0, phase ^= 1u;
            }
            src = src1, src1 = src2, xs = xs1;
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        // Nothing of this CTA's may still be in flight when it exits: each thread waits for its own
        // copies; the operator copies have landed when the phases that the loader started complete,
        // for which every producer makes up the arrivals it left out after a failed wait.
        cp_async_wait_all();
        __syncwarp();
        asm volatile("bar.sync 1, 160;" ::: "memory");   // started_items from the loader
        const int started = started_items;
        for (int k = arrived; k < started; ++k) mbar_arrive(&full_bar[k % p.nstages]);
    } else if (warp == kLoader) {
        // ------------------------------------------------------------ operator copies
        int started = 0, stage = 0;
        if (lane == 0) {
            uint32_t phase = 1;
            bool ok = true;
            for (int i = 0; i < nact && ok; ++i) {
                const F16Seg &S = seg_of(i);
                const unsigned char *w = S.w + (size_t)st.op[i] * S.w_op + (size_t)blockIdx.y * S.K * ncta * 2 * NPL;
                for (int k0 = 0; k0 < S.K; k0 += S.chunk) {
                    if (!mbar_wait(&empty_bar[stage], phase, p.wait_ns) || *(volatile int *)&abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t bytes = (uint32_t)(min(S.chunk, S.K - k0) * NPL * ncta * 2);
                    mbar_arrive_tx(&full_bar[stage], bytes);
                    bulk_g2s(base + (size_t)stage * p.stage_bytes + NPL * aplane, w + (size_t)k0 * ncta * 2 * NPL, bytes,
                             &full_bar[stage]);
                    ++started;
                    if (++stage == p.nstages) stage = 0, phase ^= 1u;
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
            for (int k = max(0, started - p.nstages); k < started; ++k)
                if (!mbar_wait(&full_bar[k % p.nstages], (k / p.nstages) & 1, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
        __syncwarp();
    } else if (warp == kIssuer || warp == kIssuer + 1) {
        // ------------------------------------------------------------ MMA issuers
        // Two warps take turns at the chunks: issuing returns only as the tensor pipe takes the products,
        // so that one warp's barrier waits (about 120 cycles each even if the phase is complete) run
        // beside the other's products.  A chunk's waits begin only when the other warp's for the chunk
        // before are over (turn_bar): the two use the stages and accumulators in turn, and a barrier's parity
        // tells a phase from the one before only once that one is known to be complete.  A segment with one
        // accumulator is one turn: its products are issued by one thread, in their order.  The whole warp runs
        // the loop, in uniform control flow and with the products unrolled, and one elected lane issues
        // (mma_f16_elected).
        const int mine = warp - kIssuer;
        int item = 0;
        const uint32_t elected = elect_one(), idesc = make_idesc(ncta, 0);
        const int n = __shfl_sync(0xffffffffu, nact, 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), sbase = smem_u32(base);
        bool ok = true;
        int stage = 0, b = 0;
        uint32_t phase = 0, aphase = 1;   // of the stage's full barrier and of the accumulator's tempty
        uint32_t turn = mine ^ 1;         // of its turn barrier (warp 0's first turn is free)
        for (int i = 0; i < n && ok; ++i) {
            const bool second = g.mode == GM_PARENT2 && i == 1;
            const int K = second ? p.s1.K : p.s0.K, chunk = second ? p.s1.chunk : p.s0.chunk;
            for (int k0 = 0; k0 < K; k0 += chunk, ++item) {
                const bool first = !p.seg_acc || k0 == 0, last = !p.seg_acc || k0 + chunk >= K;   // of its accumulator
                if (((p.seg_acc ? i : item) & 1) != mine) {   // the other warp's
                    if (++stage == p.nstages) stage = 0, phase ^= 1u;
                    if (last && ++b == kAcc) b = 0, aphase ^= 1u;
                    continue;
                }
                const bool ready = (!first || mbar_wait(&turn_bar[mine], turn, p.wait_ns)) &&
                                   mbar_wait(&full_bar[stage], phase, p.wait_ns) &&
                                   (!first || mbar_wait(&tempty_bar[b], aphase, p.wait_ns)) &&
                                   !*(volatile int *)&abort_flag;
                if (!__all_sync(0xffffffffu, ready)) {
                    ok = false;
                    break;
                }
                if (last) {
                    if (elected) mbar_arrive(&turn_bar[mine ^ 1]);
                    turn ^= 1u;
                }
                tc_fence_after();
                fence_proxy_async();   // the cp.async writes (generic proxy) -> tcgen05.mma
                const int kv = min(chunk, K - k0), ksteps = kv >> 4;
                const uint32_t sa = sbase + (uint32_t)(stage * p.stage_bytes), sb = sa + (uint32_t)(NPL * aplane);
                const uint32_t ap = (uint32_t)aplane >> 4, bp = (uint32_t)(kv * ncta * 2) >> 4;
                const uint64_t ad = NPL == 2 ? sw128_desc(sa) : sw64_desc(sa), bd = plain_desc(sb, ncta * 16);
                const uint32_t dt = tm + (uint32_t)(b * ncta);
                constexpr int kProd = NPL == 2 ? 3 : 6, kSteps = NPL == 2 ? 4 : 2;
#pragma unroll
                for (int pr = 0; pr < kProd; ++pr) {   // planes (a, b), small products first
                    const uint32_t pa = NPL == 2 ? (pr == 0) : (pr == 0 ? 2 : pr == 1 || pr == 3);
                    const uint32_t pb = NPL == 2 ? (pr == 1) : (pr == 2 ? 2 : pr == 1 || pr == 4);
#pragma unroll
                    for (int k = 0; k < kSteps; ++k)   // a K step of 16: two units
                        if (k < ksteps)
                            mma_f16_elected(dt, ad + (uint64_t)(pa * ap + k * 2),
                                            bd + (uint64_t)(pb * bp + (uint32_t)(k * 2 * ncta)), idesc, pr || k || !first ? 1u : 0u,
                                            elected);
                }
                if (elected) {
                    mma_commit(&empty_bar[stage]);
                    if (last) mma_commit(&tfull_bar[b]);
                }
                __syncwarp();
                if (++stage == p.nstages) stage = 0, phase ^= 1u;
                if (last && ++b == kAcc) b = 0, aphase ^= 1u;
            }
        }
        if (elected) {
            if (!ok) {
                atomicExch(p.err, FMM_ETIMEOUT);
                *(volatile int *)&abort_flag = 1;
            }
            // every MMA issued (also before an abort) completes before the tensor memory is freed
            mma_commit(&fin_bar[mine]);
            if (!mbar_wait(&fin_bar[mine], 0, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ drain and epilogue
        const int q = warp & 3, hf = (warp - kDrain0) >> 2;   // tensor-memory lane quarter, column half
        const int h0 = (ncta / 2 + 15) / 16 * 16;
        const int c0 = hf ? h0 : 0, nc = hf ? ncta - h0 : h0;   // its columns of the CTA's
        const int row = q * 32 + lane;
        float2 acc[kHalf / 2];
#pragma unroll
        for (int i = 0; i < kHalf / 2; ++i) acc[i] = make_float2(0.f, 0.f);
        auto val = [&](int n) { return g.alpha * (n & 1 ? acc[n / 2].y : acc[n / 2].x); };
        bool ok = true;
        const bool chunked = p.chunked;
        int slot = 0, b = 0;
        uint32_t phase = 0, fphase = 0;
        // the row's factor in segment i (its chunk c), taken while the products of the one before run
        auto factor = [&](int i, int c) {
            const float w = chunked ? __ldg(seg_of(i).ws + st.op[i] * seg_of(i).nch + c) : 1.f;
            ok = mbar_wait(&fac_bar[slot], fphase, p.wait_ns);
            const float x = fac[slot][row];
            if (++slot == kFacRing) slot = 0, fphase ^= 1u;
            return chunked ? x * w : x;
        };
        float f = nact > 0 ? factor(0, 0) : 0.f;
        ok = __all_sync(0xffffffffu, ok);   // (a wait can run out in some lanes alone)
        for (int i = 0; i < nact && ok; ++i) {
            const int nd = p.seg_acc ? 1 : seg_of(i).nch;
            for (int c = 0; c < nd; ++c) {
                ok = __all_sync(0xffffffffu, ok && mbar_wait(&tfull_bar[b], phase, p.wait_ns));
                if (!ok) break;
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * ncta + c0);
#pragma unroll
                for (int n0 = 0; n0 < kHalf; n0 += 32) {
                    if (n0 < nc) {
                        uint32_t v[32];
                        if (n0 + 32 <= kHalf && n0 + 32 <= nc) tmem_ld32(ta + n0, v);
                        else tmem_ld16(ta + n0, v);   // nc is a multiple of 16
                        tmem_wait_ld();
                        if (f != 0.f) {   // a row without a source holds stale values: not added
#pragma unroll
                            for (int e = 0; e < 32; e += 2)
                                if (n0 + e < kHalf && (e < 16 || n0 + 32 <= nc))
                                    acc[(n0 + e) / 2] =
                                        __ffma2_rn(make_float2(f, f),
                                                   make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])),
                                                   acc[(n0 + e) / 2]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty_bar[b]);
                if (++b == kAcc) b = 0, phase ^= 1u;
                if (c + 1 < nd) f = chunked ? factor(i, c + 1) : f;
                else if (i + 1 < nact) f = factor(i + 1, 0);
            }
            ok = __all_sync(0xffffffffu, ok);
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        const int bx = row < t.nrows ? box[row] : -1;
        if (ok && bx >= 0 && p.Y) {
            float *y = p.Y + (size_t)blockIdx.z * p.y_group + (size_t)bx * p.ldy + n_lo + c0;
#pragma unroll
            for (int n = 0; n < kHalf; n += 4)
                if (n < nc && n_lo + c0 + n < g.n_out)
                    *reinterpret_cast<float4 *>(y + n) =
                        make_float4(val(n), val(n + 1), val(n + 2), val(n + 3));
        }
        if (p.yp) {   // the row's planes: every drain warp passes the barriers, also after a failed wait
            // Largest entries of the row, per 64 columns, which can straddle the halves.  (They use the factors'
            // memory, since another 3 KB would cost a stage: the first barrier follows every read of a factor.)
            float(*const mx)[3][kRows] = reinterpret_cast<float(*)[3][kRows]>(&fac[0][0]);
            uint32_t m[3] = {0u, 0u, 0u};
#pragma unroll
            for (int n = 0; n < kHalf; ++n)
                if (n < nc) {
                    const uint32_t v = __float_as_uint(fabsf(val(n)));
                    const int ch = p.nys == 1 ? 0 : (c0 + n) >> 6;
#pragma unroll
                    for (int k = 0; k < 3; ++k) m[k] = max(m[k], ch == k ? v : 0u);
                }
            asm volatile("bar.sync 2, 256;" ::: "memory");
#pragma unroll
            for (int k = 0; k < 3; ++k) mx[hf][k][row] = __uint_as_float(m[k]);
            asm volatile("bar.sync 2, 256;" ::: "memory");
            float scale[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float inv;
                row_scale(max(__float_as_uint(mx[0][k][row]), __float_as_uint(mx[1][k][row])), scale[k], inv);
                // written by the thread that holds the first of the columns
                if (ok && bx >= 0 && k < p.nys && k * 64 >= c0 && k * 64 < c0 + nc) p.ys[(size_t)bx * p.nys + k] = inv;
            }
            if (ok && bx >= 0) {
                unsigned char *yp = p.yp + ((size_t)bx * p.ldyp + c0) * 2;
#pragma unroll
                for (int n = 0; n < kHalf; n += 8) {
                    if (n < nc && c0 + n < g.n_out) {
                        const int ch = p.nys == 1 ? 0 : (c0 + n) >> 6;   // 8 columns lie within one
                        const float sc = ch == 0 ? scale[0] : ch == 1 ? scale[1] : scale[2];
                        uint32_t w[NPL][4];
#pragma unroll
                        for (int e = 0; e < 8; e += 2) {
                            uint32_t ha[NPL], hb[NPL];
                            split_f16<NPL>(val(n + e) * sc, ha);
                            split_f16<NPL>(val(n + e + 1) * sc, hb);
#pragma unroll
                            for (int k = 0; k < NPL; ++k) w[k][e / 2] = ha[k] | (hb[k] << 16);
                        }
#pragma unroll
                        for (int k = 0; k < NPL; ++k)
                            *reinterpret_cast<uint4 *>(yp + k * p.yplane + n * 2) =
                                make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

// Rows list[i] (i without a list), i < nrows: the sum of `groups` partial rows x + k * x_group in
// order of k, written as FP32 (y, if not null) and as NPL planes (planes, if not null) with nsc
// scales a row: one, or one per 64 columns.  One warp per row, 512 columns at a time (complex box vectors
// have up to 976), which are read twice where a longer row has one scale; bound by memory.
template <int NPL>
__global__ void __launch_bounds__(256)
rows_planes_kernel(const float *__restrict__ x, long long x_group, int groups, int ldx, const int *__restrict__ list,
                   int nrows, int ncols, float *__restrict__ y, int ldy, unsigned char *__restrict__ planes,
                   long long plane_bytes, int ldp, float *__restrict__ inv_scale, int nsc) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= nrows) return;
    const int r = list ? list[i] : i;
    const float *xr = x + (size_t)r * ldx;
    float4 v[4];
    uint32_t m[4];   // largest entry of each v
    auto load = [&](int c0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + 4 * (lane + 32 * j);
            m[j] = 0u;
            v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c < ncols) {
                v[j] = *reinterpret_cast<const float4 *>(xr + c);
                for (int k = 1; k < groups; ++k) {
                    const float4 a = *reinterpret_cast<const float4 *>(xr + k * x_group + c);
                    v[j].x += a.x, v[j].y += a.y, v[j].z += a.z, v[j].w += a.w;
                }
                m[j] = max(max(__float_as_uint(fabsf(v[j].x)), __float_as_uint(fabsf(v[j].y))),
                           max(__float_as_uint(fabsf(v[j].z)), __float_as_uint(fabsf(v[j].w))));
            }
        }
    };
    uint32_t whole = 0u;   // largest entry of the row
    if (planes && nsc == 1)
        for (int c0 = 0; c0 < ncols; c0 += 512) {
            load(c0);
            whole = max(whole, __reduce_max_sync(0xffffffffu, max(max(m[0], m[1]), max(m[2], m[3]))));
        }
    for (int c0 = 0; c0 < ncols; c0 += 512) {
        if (!(planes && nsc == 1 && ncols <= 512)) load(c0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + 4 * (lane + 32 * j);
            if (y && c < ncols) *reinterpret_cast<float4 *>(y + (size_t)r * ldy + c) = v[j];
            if (!planes) continue;
            float scale, inv;
            // 64 columns: the lanes of one half of the warp
            const uint32_t half = __reduce_max_sync(lane < 16 ? 0x0000ffffu : 0xffff0000u, m[j]);
            row_scale(nsc == 1 ? whole : half, scale, inv);
            if (c >= ncols) continue;
            if (nsc == 1 ? c == 0 : (lane & 15) == 0) inv_scale[(size_t)r * nsc + (nsc == 1 ? 0 : c / 64)] = inv;
            uint32_t h[4][NPL];
            split_f16<NPL>(v[j].x * scale, h[0]), split_f16<NPL>(v[j].y * scale, h[1]);
            split_f16<NPL>(v[j].z * scale, h[2]), split_f16<NPL>(v[j].w * scale, h[3]);
#pragma unroll
            for (int k = 0; k < NPL; ++k)
                *reinterpret_cast<uint2 *>(planes + k * plane_bytes + ((size_t)r * ldp + c) * 2) =
                    make_uint2(h[0][k] | (h[1][k] << 16), h[2][k] | (h[3][k] << 16));
        }
    }
}

// Operator k (block k): rows x cols FP64, row-major, into the stage form [nsplit][chunk][plane]
// [unit][ncta rows][16 B] of the padded (nsplit * ncta) x K operator, and its 1 / scale: one for the
// operator, or (by_chunk) one per chunk.
template <int NPL>
__global__ void __launch_bounds__(256)
pack_kernel(const double *__restrict__ w, int rows, int cols, int ncta, int nsplit, int K, int chunk,
            int by_chunk, unsigned char *__restrict__ out, float *__restrict__ inv_scale) {
    __shared__ double red[256], scale[kMaxChunks];
    const double *a = w + (size_t)blockIdx.x * rows * cols;
    const int nch = (K + chunk - 1) / chunk;
    for (int c = 0; c < nch; ++c) {
        const int k0 = by_chunk ? c * chunk : 0, kn = by_chunk ? min(chunk, cols - k0) : cols;
        double m = 0;
        for (int i = threadIdx.x; i < rows * kn; i += 256) m = fmax(m, fabs(a[(size_t)(i / kn) * cols + k0 + i % kn]));
        red[threadIdx.x] = m;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            int ex = 0;
            frexp(red[0], &ex);
            scale[c] = red[0] > 0 ? ldexp(1.0, 14 - ex) : 1.0;
            if (by_chunk || c == 0)
                inv_scale[by_chunk ? blockIdx.x * nch + c : blockIdx.x] = red[0] > 0 ? (float)ldexp(1.0, ex - 14) : 0.f;
        }
        __syncthreads();
    }
    const int total = nsplit * ncta * K;
    unsigned char *o = out + (size_t)blockIdx.x * total * 2 * NPL;
    for (int i = threadIdx.x; i < total; i += 256) {
        const int n = i / K, k = i % K;                 // output row, input column
        const int ns = n / ncta, r = n % ncta, c = k / chunk, kin = k % chunk;
        const int kv = min(chunk, K - c * chunk);
        double x = n < rows && k < cols ? a[(size_t)n * cols + k] * scale[c] : 0.0;
        const size_t off = ((size_t)ns * K + (size_t)c * chunk) * ncta * 2 * NPL + ((size_t)(kin >> 3) * ncta + r) * 16 +
                           (kin & 7) * 2;
        for (int pl = 0; pl < NPL; ++pl) {
            const __half h = __float2half_rn((float)x);
            x -= (double)__half2float(h);
            *reinterpret_cast<__half *>(o + off + (size_t)pl * kv * ncta * 2) = h;
        }
    }
}

// Two planes: 64 values of K a chunk, the columns of a scale.  Three: at most 32, evened out.
int chunk_of(int K, int planes) {
    if (planes == 2) return 64;
    const int n = (K + 31) / 32;
    return round_up((K + n - 1) / n, 16);
}

}  // namespace

// Groups that the 189 transfer vectors of a level's stencil are cut into.  A tile walks its active
// vectors one after the other (about 1 us each), so a level with few tiles leaves most SMs idle for
// as long as one tile takes: levels 2 and 3 have at most 8 tiles (one a class), level 4 8 to 32 and
// level 5 16 to 256.  The groups' partial rows are added in order, so a result does not depend on how
// many CTAs there are, and the number depends on the level alone: the same boxes give the same bits in
// any partition.  Step of 20k points (FP32, depth 3), Helmholtz evaluation (131k, depth 4), FP64 (100k,
// depth 4): 359, 809, 10083 us; half as many groups 358, 819, 10198; twice as many 359, 834, 10090; none
// 506, 1063, 10342.
int stencil_groups(const OpSet &o, int level) {
    // Real FP16X3 sums stay one sequence a box.  With charges of one sign a potential is 2^depth times its
    // variation across a leaf, so that gradients carry the rounding of the sums (cube, p = 6: 2.3e-5 at depth 5,
    // 4.7e-5 at depth 6, against FP64); another order of the same sums is no less exact, but gives gradients
    // that differ by as much (2.2e-5 and 4.6e-5).  Sums of complex densities differ by 3e-6 at most
    // (depths 2 to 5).
    if (!o.cplx && o.f_stencil.planes == 2) return 1;
    return level <= 3 ? 19 : level == 4 ? 9 : level == 5 ? 7 : 1;
}

cudaError_t f16_upload(fmm_ctx *ctx, const double *w, int count, int rows, int cols, int K, int planes,
                       bool chunk_scales, F16Mat *out) {
    out->K = K, out->planes = planes;
    const int np = round_up(rows, 16);
    out->nsplit = (np + kMaxCols - 1) / kMaxCols;
    out->ncta = round_up((np + out->nsplit - 1) / out->nsplit, 16);
    out->chunk = chunk_of(K, planes);
    out->op_bytes = (size_t)out->nsplit * out->ncta * K * 2 * planes;
    void *d = nullptr, *ds = nullptr, *src = nullptr;
    FMM_CUDA_TRY(dev_malloc(&d, out->op_bytes * count));
    ctx->op_allocs.push_back(d);
    const int nch = (K + out->chunk - 1) / out->chunk;
    if (nch > kMaxChunks) return cudaErrorInvalidValue;
    FMM_CUDA_TRY(dev_malloc(&ds, (size_t)count * nch * sizeof(float)));
    ctx->op_allocs.push_back(ds);
    const size_t n = (size_t)count * rows * cols * sizeof(double);
    cudaStream_t s = ctx->stream;
    Scratch<double> tmp;
    FMM_CUDA_TRY(tmp.alloc((size_t)count * rows * cols, s));
    src = tmp.p;
    FMM_CUDA_TRY(cudaMemcpyAsync(src, w, n, cudaMemcpyHostToDevice, s));
    auto go = [&](auto kern) {
        kern<<<count, 256, 0, s>>>((const double *)src, rows, cols, out->ncta, out->nsplit, K, out->chunk, chunk_scales,
                                   (unsigned char *)d, (float *)ds);
    };
    planes == 2 ? go(pack_kernel<2>) : go(pack_kernel<3>);
    count_launch();
    FMM_CUDA_TRY(cudaGetLastError());
    FMM_CUDA_TRY(cudaStreamSynchronize(s));   // the host operators may be released
    out->data = d, out->scale = (float *)ds;
    return cudaSuccess;
}

cudaError_t launch_rows_planes(const float *x, long long x_group, int groups, int ldx, const int *list, int64_t nrows,
                               int ncols, float *y, int ldy, void *planes, long long plane_bytes, int ldp,
                               float *inv_scale, int nsc, int nplanes, cudaStream_t s) {
    if (nrows <= 0) return cudaSuccess;
    if (nsc != 1 && nsc != (ncols + 63) / 64) return cudaErrorInvalidValue;
    if (ncols & 15) return cudaErrorInvalidValue;
    auto go = [&](auto kern) {
        kern<<<(unsigned)((nrows + 7) / 8), 256, 0, s>>>(x, x_group, groups, ldx, list, (int)nrows, ncols, y, ldy,
                                                         (unsigned char *)planes, plane_bytes, ldp, inv_scale, nsc);
    };
    nplanes == 2 ? go(rows_planes_kernel<2>) : go(rows_planes_kernel<3>);
    count_launch();
    return cudaGetLastError();
}

GemmDev make_gemm_dev(const fmm_ctx *ctx, const GemmCall &c);

cudaError_t gemm_f16(const fmm_ctx *ctx, const GemmCall &c, const F16Mat &W, const F16Mat *W1, cudaStream_t s) {
    F16Dev p{};
    p.g = make_gemm_dev(ctx, c);
    const bool cls = c.mode == GM_STENCIL || c.mode == GM_PARENT2;
    const TileSet &ts = c.tiles ? *c.tiles : cls ? ctx->tiles_cls[c.level] : ctx->tiles_plain[c.level];
    if (ts.ntiles == 0) return cudaSuccess;
    p.g.tiles = ts.tiles;
    p.g.masks = ts.masks;
    if (c.mode == GM_STENCIL && ctx->masks_ev) FMM_CUDA_TRY(cudaStreamWaitEvent(s, ctx->masks_ev, 0));
    auto seg = [&](const void *xp, long long plane, int ld, const float *xs, const F16Mat &m) {
        F16Seg q{};
        q.xp = (const unsigned char *)xp, q.xplane = plane, q.ld = ld, q.xs = xs;
        q.w = (const unsigned char *)m.data, q.w_op = (long long)m.op_bytes, q.ws = m.scale;
        q.K = m.K, q.chunk = m.chunk, q.nch = (m.K + m.chunk - 1) / m.chunk;
        q.nxs = c.xp_chunk_scales ? q.nch : 1;
        return q;
    };
    p.s0 = p.s1 = seg(c.Xp, c.xp_plane, c.xp_ld, c.xp_scale, W);
    if (c.mode == GM_PARENT2 && c.X1) {
        if (!W1 || W1->ncta != W.ncta || W1->nsplit != W.nsplit || W1->planes != W.planes) return cudaErrorInvalidValue;
        p.s1 = seg(c.Xp1, c.xp1_plane, c.xp1_ld, c.xp1_scale, *W1);
    }
    for (const F16Seg *q : {&p.s0, &p.s1})
        if (!q->xp || !q->xs || !q->w || ((uintptr_t)q->xp & 15) || (q->xplane & 15) || (q->ld & 7) || (q->K & 15) ||
            q->K > q->ld)
            return cudaErrorInvalidValue;
    const int npl = W.planes;
    p.ncta = W.ncta;
    p.stage_bytes = round_up((kRows * (npl == 2 ? kRowBytes<2> : kRowBytes<3>) +
                              std::max(p.s0.chunk, p.s1.chunk) * W.ncta * 2) * npl, 1024);
    auto kern = npl == 2 ? gemm_f16_kernel<2> : gemm_f16_kernel<3>;
    int most = 0;
    FMM_CUDA_TRY(allow_all_shared(kern, &most));
    p.nstages = std::min(kMaxStages, (most - 1024) / p.stage_bytes);
    if (p.nstages < 2) return cudaErrorInvalidValue;
    int cols = 32;
    while (cols < kAcc * p.ncta) cols <<= 1;
    if (cols > 512) return cudaErrorInvalidValue;
    p.tmem_cols = cols;
    p.groups = c.groups;
    p.chunked = c.xp_chunk_scales;
    p.seg_acc = c.mode == GM_STENCIL && npl == 2 && !c.xp_chunk_scales;
    p.Y = (float *)c.Y, p.ldy = c.ldy, p.y_group = c.y_group;
    if (c.Yp) {
        if (W.nsplit != 1 || c.groups != 1 || !c.yp_scale) return cudaErrorInvalidValue;
        p.yp = (unsigned char *)c.Yp, p.yplane = c.yp_plane, p.ldyp = c.yp_ld, p.ys = c.yp_scale;
        p.nys = c.yp_chunk_scales ? (c.n_out + 63) / 64 : 1;
    }
    p.err = ctx->dev_flag;
    p.wait_ns = ctx->tc_wait_ns;
    const size_t smem = (size_t)p.nstages * p.stage_bytes + 1024;
    kern<<<dim3(ts.ntiles, W.nsplit, c.groups), kThreads, smem, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

}  // namespace fmm
