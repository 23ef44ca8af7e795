// Tensor-core (tcgen05, sm_103a) form of the gathered GEMM of gemm_common.cuh, with split-
// precision operands: the FP32 inputs are split into BF16 (hi, lo[, mid]) or TF32 (big, small)
// planes and the products a_i b_j with i + j below the split order are accumulated in FP32 in
// tensor memory.  This carries the surface contractions and the M2L (VLI) of the FMM.
//
// Layout.  One CTA computes a 128-row tile (M = 128 boxes) for all N output columns.  The K
// dimension of every segment is cut into chunks of one 128-byte swizzle atom (64 BF16 or 32
// TF32 values).  A stage holds the A planes (128 rows x 128 B each, K-major, SWIZZLE_128B:
// 16-byte unit j of row r sits at (j ^ (r % 8)) * 16 within the row's 128 bytes, rows 128 B
// apart, 8-row groups 1024 B apart) and the B planes (N rows, same layout).  B (the operator) is
// stored in global memory already in this layout, chunk by chunk, so one bulk copy per stage
// moves it; A rows are gathered by the producer warps, split and written with st.shared.
//
// Warp roles (256 threads, two warps per SM sub-partition so that the accumulator warps can hold
// 160 FP32 partial sums in registers): warps 4-7 drain the tensor memory accumulators (warp w
// owns TMEM lanes 32(w-4).. = tile rows) into FP32 registers and write Y; warp 0 owns the tensor
// memory allocation.  A rows from FP32 (gathered and split in registers): warps 0-3 produce the
// stages and lane 0 of warp 4 issues every tcgen05.mma (item i), after which its warp drains item
// i - 1.  A rows from split planes (copies only): warps 0-2 produce and lane 0 of warp 3 issues,
// so the tensor pipe keeps running while all four accumulator warps drain (issuing an item's
// MMAs takes as long as the tensor pipe needs for them).
//
// Accumulation.  The tensor core adds an MMA's products into the FP32 accumulator with
// truncation, so a long chain of MMAs into one accumulator drifts toward zero by about one
// half-ulp per step.  Every stage (at most 4 k-steps x the split products) therefore gets a
// fresh accumulator (two alternate in tensor memory) and its partial sum is added, correctly
// rounded, into registers of the accumulator warps.  A CTA covers at most 160 output columns;
// wider outputs are split over blockIdx.y.
//
// Every mbarrier wait is bounded (1 s of %globaltimer); on expiry the kernel records an error
// code in a device flag, stops producing/issuing, still releases its tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gemm_common.cuh"
#include "tcgen05.cuh"

namespace fmm {

constexpr int kTcThreads = 256;           // 4 producer warps, 4 accumulator warps (one issues MMAs)
constexpr int kTcRows = 128;
constexpr int kTcMaxN = 160;               // output columns per CTA (wider N: several CTAs)
constexpr int kAtomBytes = 128;            // one swizzle atom row
constexpr int kPlaneProducers = 96;        // plane mode: warps 0-2 copy, warp 3 issues the MMAs
constexpr int kPlaneStages = 2;            // plane mode: stages in shared memory

struct TcDev {
    GemmDev g;                      // gather description (W fields unused)
    const unsigned char *Wt0;       // tensor-core operand of segment 0 (or of segment index * stride)
    long long wt_stride;            // bytes between consecutive operators (CHILDREN, STENCIL)
    const unsigned char *Wt1[8];    // PARENT2 segment 1 by class
    int nplanes;                    // 2 (x3) or 3 (x6)
    int tf32;                       // 1: kind::tf32 planes (4-byte); 0: BF16 planes (2-byte)
    int nprod;                      // products per k-step
    int prod_a[6], prod_b[6];       // plane pairs
    int nstages;
    int ncta;                       // output columns per CTA (grid.y splits wider N)
    int tmem_cols;
    int *err;                       // device error flag
    unsigned long long wait_ns;     // bound on every pipeline barrier wait (default 1 s)
    int a_planes;                   // A rows arrive pre-split from xp (cp.async copies)
    const unsigned char *xp;        // split planes of the A rows
    long long xp_plane;             // bytes between planes
    int xp_ld;                      // row stride in elements
    unsigned char *yp;              // split-plane output (instead of FP32 Y) if non-null
    long long yp_plane;             // bytes between output planes
    int yp_ld;                      // output row stride in elements
};

namespace {

// ---------------------------------------------------------------- splits
__device__ __forceinline__ uint32_t bf16_bits(float x) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}
__device__ __forceinline__ float bf16_val(uint32_t b) {
    return __bfloat162float(__ushort_as_bfloat16((unsigned short)b));
}
__device__ __forceinline__ uint32_t tf32_round(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r & 0xffffe000u;   // keep the 10 explicit mantissa bits only
}

// Teardown: wait (at most 1 s each) until the operator copies this thread started have landed,
// so that no copy is still writing into shared memory when the CTA exits, also after an abort.
__device__ __forceinline__ bool wait_bulk_copies(uint64_t *bulk_bar, const int *started, int nstages) {
    bool ok = true;
    for (int s = 0; s < nstages; ++s)
        if (started[s] > 0) ok = mbar_wait(&bulk_bar[s], (uint32_t)(started[s] - 1) & 1u, kWaitNs) && ok;
    return ok;
}

// ---------------------------------------------------------------- work list helpers
struct SegInfo {
    const float *X;
    int ldx, K;
    const unsigned char *Wt;
    int nchunks;
};

// Per-tile tables held in shared memory: the operator index and the transfer vector of every
// class slot of the tile's octant class (stencil mode), so that moving to the next segment
// needs no dependent global loads.
struct TileTables {
    int slot[kClassSlots];
    int delta[kClassSlots];
};

__device__ __forceinline__ long long w_index_fast(const GemmDev &g, const Tile &t, const TileTables &tt, int seg) {
    return g.mode == GM_STENCIL ? (long long)tt.slot[seg] : gemm_w_index(g, t, seg);
}

__device__ __forceinline__ SegInfo seg_info(const TcDev &p, const Tile &t, const TileTables &tt, int seg,
                                            int chunk_elems) {
    SegInfo s;
    const GemmDev &g = p.g;
    const bool second = g.mode == GM_PARENT2 && seg == 1;
    s.X = (const float *)(second ? g.X1 : g.X0);
    s.ldx = second ? g.ldx1 : g.ldx0;
    s.K = second ? g.k1 : g.k0;
    s.Wt = second ? p.Wt1[t.cls] : p.Wt0 + w_index_fast(g, t, tt, seg) * p.wt_stride;
    s.nchunks = (s.K + chunk_elems - 1) / chunk_elems;
    return s;
}

// One tile row: its box and, for the stencil, the box's integer coordinates.
struct RowRef {
    int box, ax, ay, az;
};

__device__ __forceinline__ RowRef row_ref(const GemmDev &g, int box) {
    RowRef r{box, 0, 0, 0};
    if (box >= 0 && g.mode == GM_STENCIL) demorton3(g.keys[box], r.ax, r.ay, r.az);
    return r;
}

// source row of (row, seg), -1 for none (one global load: the dense table or the child/parent table)
__device__ __forceinline__ int src_fast(const GemmDev &g, const Tile &t, const TileTables &tt, const RowRef &r,
                                        int seg) {
    if (r.box < 0) return -1;
    if (g.mode == GM_STENCIL) {
        int dx, dy, dz;
        unpack_delta(tt.delta[seg], dx, dy, dz);
        return dense_find(g.dense, g.level, r.ax + dx, r.ay + dy, r.az + dz);
    }
    return gemm_src_row(g, t, r.box, seg);
}


}  // namespace

// The kernel body.  PL (plane layout, A rows from split planes): 384 threads, warps 0-2
// produce, warp 3 issues, warps 4-11 drain, two per TMEM lane quarter, each holding half of the
// row's columns (80), so that a CTA needs about half the registers of the 256-thread layout and
// near-field CTAs can share its SM.  Otherwise: 256 threads, warps 0-3 gather and split A in
// registers, warps 4-7 drain whole rows (warp 4 also issues).
template <bool TF32, bool PL>
__device__ __forceinline__ void tc_body(const TcDev &p) {
    constexpr int NT = PL ? 384 : kTcThreads;        // threads
    constexpr int DC = PL ? kTcMaxN / 2 : kTcMaxN;   // columns a drain thread holds
    constexpr int NDRAIN = PL ? 8 : 4;               // drain warps
    extern __shared__ unsigned char smem_raw[];
    // full: the producers' A rows of a stage; bulk: its operator copy; empty: the stage's MMAs
    // done; tfull / tempty: an accumulator's MMAs done / drained; fin: every MMA of the CTA done
    __shared__ uint64_t full_bar[4], bulk_bar[4], empty_bar[4], tfull_bar[2], tempty_bar[2], fin_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int box[kTcRows];
    __shared__ int srcs[2][kTcRows];
    __shared__ uint32_t mask[6];
    __shared__ int abort_flag;
    __shared__ TileTables tt;

    const GemmDev &g = p.g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Tile t = g.tiles[blockIdx.x];
    const int n_lo = blockIdx.y * p.ncta;                 // this CTA's output columns
    const int N = min(p.ncta, g.n_out - n_lo);            // multiple of 16
    constexpr int esz = TF32 ? 4 : 2;                     // bytes per plane element
    constexpr int chunk_elems = kAtomBytes / esz;         // K values per stage
    const int a_plane_bytes = kTcRows * kAtomBytes;       // 16 KB
    const int b_plane_bytes = N * kAtomBytes;
    const int stage_bytes = p.nplanes * (a_plane_bytes + p.ncta * kAtomBytes);
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

    if (tid == 0) {
        for (int s = 0; s < p.nstages; ++s) {
            // register gather: 4 producer warps; plane copies: 96 cp.async arrivals (3 producer warps)
            mbar_init(&full_bar[s], p.a_planes ? kPlaneProducers : 4);
            mbar_init(&bulk_bar[s], 1);       // thread 0's expect_tx arrive, then the copy's bytes
            mbar_init(&empty_bar[s], 1);      // tcgen05.commit
        }
        mbar_init(&fin_bar, 1);               // tcgen05.commit after the last MMA
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull_bar[b], 1);      // tcgen05.commit
            mbar_init(&tempty_bar[b], NDRAIN);   // the accumulator warps
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 6) mask[tid] = g.mode == GM_STENCIL ? g.masks[(size_t)t.mask * 6 + tid] : 0xffffffffu;
    if (tid < kTcRows) box[tid] = tid < t.nrows ? gemm_row_box(g, t, tid) : -1;
    if (g.mode == GM_STENCIL)
        for (int k = tid; k < kClassSlots; k += NT) {
            tt.slot[k] = g.class_slots[t.cls * kClassSlots + k];
            tt.delta[k] = g.class_delta[t.cls * kClassSlots + k];
        }
    if (warp == 0) tmem_alloc(&tmem_base, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    const uint32_t idesc = make_idesc(N, TF32 ? 2 : 1);
    const int nseg = gemm_nseg(g);
    auto active = [&](int seg) { return g.mode != GM_STENCIL || ((mask[seg >> 5] >> (seg & 31)) & 1u); };
    // number of stage items (segment chunks) of the tile
    int n_items = 0;
    for (int seg = 0; seg < nseg; ++seg)
        if (active(seg)) n_items += (gemm_seg_k(g, seg) + chunk_elems - 1) / chunk_elems;
    // the split products (plane pairs), held in registers
    int pa[6], pb[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) pa[i] = p.prod_a[i], pb[i] = p.prod_b[i];

    // One stage item's MMAs into accumulator b, issued by one thread: the split products of the
    // chunk, then commits that free the stage and mark the accumulator full.
    auto issue_item = [&](int stage, int b, const SegInfo &si, int chunk) {
        tc_fence_after();
        fence_proxy_async();   // cp.async / st.shared writes (generic proxy) -> tcgen05.mma
        const uint32_t sa = smem_u32(base + (size_t)stage * stage_bytes);
        const uint32_t sb = sa + p.nplanes * a_plane_bytes;
        const uint32_t dt = tmem + (uint32_t)(b * p.ncta);
        const int kval = min(chunk_elems, si.K - chunk * chunk_elems);
        const int ksteps = min(kAtomBytes / 32, (kval * esz + 31) / 32);
        // descriptors of the stage's planes; a K step of 32 bytes adds 2 to the address field
        const uint64_t a0 = sw128_desc(sa), b0 = sw128_desc(sb);
        uint32_t accum = 0u;
#pragma unroll
        for (int pr = 0; pr < 6; ++pr) {
            if (pr >= p.nprod) break;
            const uint64_t ap = a0 + (uint64_t)((pa[pr] * a_plane_bytes) >> 4);
            const uint64_t bp = b0 + (uint64_t)((pb[pr] * b_plane_bytes) >> 4);
            for (int ks = 0; ks < ksteps; ++ks) {
                if (TF32) mma_tf32(dt, ap + 2 * ks, bp + 2 * ks, idesc, accum);
                else mma_f16(dt, ap + 2 * ks, bp + 2 * ks, idesc, accum);
                accum = 1;
            }
        }
        mma_commit(&empty_bar[stage]);
        mma_commit(&tfull_bar[b]);
    };

    if (warp < 3 && p.a_planes) {
        // ------------------------------------------------------------ producers, split planes
        // The source rows are already split into planes in global memory, so the producers only
        // copy: every thread issues 16-byte cp.async copies straight into the swizzled stage
        // (8 lanes per row, 4 rows per warp instruction, zero fill for missing rows), then
        // arrives on the stage barrier when its copies have landed.
        // Thread 0 adds the operator's bulk copy.  Copies of several stages stay in flight.
        // Every producer thread runs the same segment loop and the same named barrier per active
        // segment whatever happens; after a failed (bounded) wait it only skips its copies.
        // The source row of the next active segment is looked up while the current one is copied.
        // Three warps (96 threads) cover the 128 rows: thread i looks up rows i and i + 96.
        int item = 0, sidx = 0;
        int bulk_started[4] = {0, 0, 0, 0};   // operator copies thread 0 started per stage
        bool ok = true;
        const bool two = tid + kPlaneProducers < kTcRows;
        const RowRef me = row_ref(g, box[tid]);
        const RowRef me2 = row_ref(g, two ? box[tid + kPlaneProducers] : -1);
        int seg = 0;
        while (seg < nseg && !active(seg)) ++seg;
        int src_next = seg < nseg ? src_fast(g, t, tt, me, seg) : -1;
        int src_next2 = seg < nseg ? src_fast(g, t, tt, me2, seg) : -1;
        for (; seg < nseg;) {
            int seg2 = seg + 1;
            while (seg2 < nseg && !active(seg2)) ++seg2;
            const SegInfo si = seg_info(p, t, tt, seg, chunk_elems);
            srcs[sidx][tid] = src_next;
            if (two) srcs[sidx][tid + kPlaneProducers] = src_next2;
            asm volatile("bar.sync 1, 96;" ::: "memory");
            src_next = seg2 < nseg ? src_fast(g, t, tt, me, seg2) : -1;
            src_next2 = seg2 < nseg ? src_fast(g, t, tt, me2, seg2) : -1;
            const int *rs = srcs[sidx];
            const int unit = lane & 7;
            for (int c = 0; c < si.nchunks; ++c, ++item) {
                const int stage = item % p.nstages;
                if (!ok) continue;
                if ((item >= p.nstages && !mbar_wait(&empty_bar[stage], ((item / p.nstages) - 1) & 1, p.wait_ns)) ||
                    *(volatile int *)&abort_flag) {
                    ok = false;
                    continue;
                }
                unsigned char *sa = base + (size_t)stage * stage_bytes;
                unsigned char *sb = sa + p.nplanes * a_plane_bytes;
                if (tid == 0) {
                    mbar_arrive_tx(&bulk_bar[stage], (uint32_t)(p.nplanes * b_plane_bytes));
                    ++bulk_started[stage];
                    const size_t plane_full = (size_t)g.n_out * kAtomBytes;
                    if ((size_t)b_plane_bytes == plane_full)   // the chunk's planes are contiguous: one copy
                        bulk_g2s(sb, si.Wt + (size_t)c * p.nplanes * plane_full,
                                 (uint32_t)(p.nplanes * b_plane_bytes), &bulk_bar[stage]);
                    else
                        for (int pl = 0; pl < p.nplanes; ++pl)
                            bulk_g2s(sb + pl * b_plane_bytes,
                                     si.Wt + ((size_t)c * p.nplanes + pl) * plane_full + (size_t)n_lo * kAtomBytes,
                                     (uint32_t)b_plane_bytes, &bulk_bar[stage]);
                }
                const int k0 = c * chunk_elems;
                const int kval = min(chunk_elems, si.K - k0);
                const int valid_units = (kval * esz + 15) / 16;
                const bool unit_ok = unit < valid_units;
#pragma unroll
                for (int j = 0; j < (kTcRows + 11) / 12; ++j) {   // 12 rows per pass of 3 warps
                    const int r = j * 12 + warp * 4 + (lane >> 3);
                    if (r >= kTcRows) break;
                    const int sr = rs[r];
                    const bool have = unit_ok && sr >= 0;
                    if (!unit_ok) continue;   // K units past the segment are never read
                    const size_t elem = (size_t)(have ? sr : 0) * p.xp_ld + k0 + unit * (16 / esz);
                    const int dst_off = r * kAtomBytes + ((unit ^ (r & 7)) << 4);
#pragma unroll
                    for (int pl = 0; pl < 3; ++pl) {
                        if (pl < p.nplanes)
                            cp_async16(sa + pl * a_plane_bytes + dst_off, p.xp + pl * p.xp_plane + elem * esz,
                                       have ? 16 : 0);
                    }
                }
                cp_async_arrive(&full_bar[stage]);
            }
            sidx ^= 1;
            seg = seg2;
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        // nothing of this thread's may still be in flight when the CTA exits
        cp_async_wait_all();
        if (tid == 0 && !wait_bulk_copies(bulk_bar, bulk_started, p.nstages)) atomicExch(p.err, FMM_ETIMEOUT);
    } else if (warp == 3 && p.a_planes) {
        // ------------------------------------------------------------ MMA issuer (plane mode)
        // A warp of its own issues the MMAs, so the tensor pipe runs while the accumulator
        // warps drain: the issue of an item's MMAs returns only as the tensor pipe takes them.
        if (lane == 0) {
            bool ok = true;
            int seg = 0, chunk = 0;
            while (seg < nseg && !active(seg)) ++seg;
            SegInfo si{};
            if (seg < nseg) si = seg_info(p, t, tt, seg, chunk_elems);
            for (int item = 0; item < n_items; ++item) {
                const int stage = item % p.nstages, b = item & 1;
                if (!mbar_wait(&full_bar[stage], (item / p.nstages) & 1, p.wait_ns) ||
                    !mbar_wait(&bulk_bar[stage], (item / p.nstages) & 1, p.wait_ns) ||
                    (item >= 2 && !mbar_wait(&tempty_bar[b], ((item >> 1) - 1) & 1, p.wait_ns)) ||
                    *(volatile int *)&abort_flag) {
                    ok = false;
                    break;
                }
                issue_item(stage, b, si, chunk);
                if (++chunk == si.nchunks) {
                    chunk = 0;
                    ++seg;
                    while (seg < nseg && !active(seg)) ++seg;
                    if (seg < nseg) si = seg_info(p, t, tt, seg, chunk_elems);
                }
            }
            if (!ok) {
                atomicExch(p.err, FMM_ETIMEOUT);
                *(volatile int *)&abort_flag = 1;
            }
            // every MMA issued (also before an abort) completes before the tensor memory is freed
            mma_commit(&fin_bar);
            if (!mbar_wait(&fin_bar, 0, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
        }
    } else if (!PL && warp < 4) {
        // ------------------------------------------------------------ producers
        int item = 0;
        int bulk_started[4] = {0, 0, 0, 0};   // operator copies thread 0 started per stage
        bool ok = true;
        const RowRef me = row_ref(g, box[tid]);
        int seg0 = 0;
        while (seg0 < nseg && !active(seg0)) ++seg0;
        int src_next = seg0 < nseg ? src_fast(g, t, tt, me, seg0) : -1;
        for (int seg = seg0; seg < nseg && ok;) {
            int seg2 = seg + 1;
            while (seg2 < nseg && !active(seg2)) ++seg2;
            const SegInfo si = seg_info(p, t, tt, seg, chunk_elems);
            // source row of this warp's rows (row 32 * warp + lane), shared by shuffles; the
            // next segment's is looked up now
            const int my_src = src_next;
            src_next = seg2 < nseg ? src_fast(g, t, tt, me, seg2) : -1;
            for (int c = 0; c < si.nchunks; ++c, ++item) {
                const int stage = item % p.nstages;
                if (item >= p.nstages && !mbar_wait(&empty_bar[stage], ((item / p.nstages) - 1) & 1, p.wait_ns)) {
                    ok = false;
                    break;
                }
                if (*(volatile int *)&abort_flag) { ok = false; break; }
                unsigned char *sa = base + (size_t)stage * stage_bytes;
                unsigned char *sb = sa + p.nplanes * a_plane_bytes;
                if (tid == 0) {
                    // rows [n_lo, n_lo + N) of every plane of chunk c: contiguous per plane, and
                    // all planes contiguous when the CTA covers every row (one copy then)
                    mbar_arrive_tx(&bulk_bar[stage], (uint32_t)(p.nplanes * b_plane_bytes));
                    ++bulk_started[stage];
                    const size_t plane_full = (size_t)g.n_out * kAtomBytes;
                    if ((size_t)b_plane_bytes == plane_full)
                        bulk_g2s(sb, si.Wt + (size_t)c * p.nplanes * plane_full,
                                 (uint32_t)(p.nplanes * b_plane_bytes), &bulk_bar[stage]);
                    else
                        for (int pl = 0; pl < p.nplanes; ++pl)
                            bulk_g2s(sb + pl * b_plane_bytes,
                                     si.Wt + ((size_t)c * p.nplanes + pl) * plane_full + (size_t)n_lo * kAtomBytes,
                                     (uint32_t)b_plane_bytes, &bulk_bar[stage]);
                }
                // gather: each warp covers its 32 rows; lanes split a row into 16-byte pieces.
                // All loads of the warp are issued before any is used (memory-level parallelism).
                const int k0 = c * chunk_elems;
                const int kval = min(chunk_elems, si.K - k0);       // valid K values in this chunk
                constexpr int per_row = chunk_elems / 4;            // float4 loads per row
                constexpr int rows_per_pass = 32 / per_row;
                constexpr int passes = 32 / rows_per_pass;
                const int my_row_in_pass = lane / per_row, my_q = lane % per_row;
                const int k = my_q * 4;                             // first of 4 values
                float4 vbuf[passes];
#pragma unroll
                for (int ps = 0; ps < passes; ++ps) {
                    const int r = warp * 32 + ps * rows_per_pass + my_row_in_pass;
                    const int sr = __shfl_sync(0xffffffffu, my_src, r - warp * 32);
                    vbuf[ps] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (sr >= 0 && k < kval)
                        vbuf[ps] = __ldg(reinterpret_cast<const float4 *>(si.X + (size_t)sr * si.ldx + k0 + k));
                }
#pragma unroll
                for (int ps = 0; ps < passes; ++ps) {
                    const int r = warp * 32 + ps * rows_per_pass + my_row_in_pass;
                    const float x[4] = {vbuf[ps].x, vbuf[ps].y, vbuf[ps].z, vbuf[ps].w};
                    const int rowoff = (r >> 3) * 1024 + (r & 7) * 128;
                    if (!TF32) {
                        // 4 BF16 values = 8 bytes: half of a 16-byte unit
                        const int unit = k >> 3, half = (k >> 2) & 1;
                        const int off = rowoff + ((unit ^ (r & 7)) << 4) + half * 8;
                        uint32_t hb[4], lb[4], mb[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            hb[i] = bf16_bits(x[i]);
                            const float r1 = x[i] - bf16_val(hb[i]);
                            lb[i] = bf16_bits(r1);
                            mb[i] = bf16_bits(r1 - bf16_val(lb[i]));
                        }
                        // plane order: 0 = hi, 1 = lo, 2 = third term
                        *reinterpret_cast<uint2 *>(sa + off) = make_uint2(hb[0] | (hb[1] << 16), hb[2] | (hb[3] << 16));
                        *reinterpret_cast<uint2 *>(sa + a_plane_bytes + off) =
                            make_uint2(lb[0] | (lb[1] << 16), lb[2] | (lb[3] << 16));
                        if (p.nplanes == 3)
                            *reinterpret_cast<uint2 *>(sa + 2 * a_plane_bytes + off) =
                                make_uint2(mb[0] | (mb[1] << 16), mb[2] | (mb[3] << 16));
                    } else {
                        // 4 TF32 values = one 16-byte unit
                        const int unit = k >> 2;
                        const int off = rowoff + ((unit ^ (r & 7)) << 4);
                        uint32_t bb[4], ss[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            bb[i] = tf32_round(x[i]);
                            ss[i] = tf32_round(x[i] - __uint_as_float(bb[i]));
                        }
                        *reinterpret_cast<uint4 *>(sa + off) = make_uint4(bb[0], bb[1], bb[2], bb[3]);
                        *reinterpret_cast<uint4 *>(sa + a_plane_bytes + off) = make_uint4(ss[0], ss[1], ss[2], ss[3]);
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_bar[stage]);
            }
            seg = seg2;
        }
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        }
        if (tid == 0 && !wait_bulk_copies(bulk_bar, bulk_started, p.nstages)) atomicExch(p.err, FMM_ETIMEOUT);
    } else {
        // ------------------------------------------------------------ accumulators / epilogue
        // Each stage item's products land in one of two TMEM accumulators; these warps add the
        // item's partial sums (32 rows each) into FP32 registers, so that no TMEM accumulator
        // takes more than one stage of tensor-core additions.
        const int q = (warp - 4) & 3;                     // TMEM lane quarter
        const int hf = PL ? (warp - 4) >> 2 : 0;          // column half (PL)
        const int c0 = hf * DC;                           // first column this thread holds
        const bool issuer = !PL && warp == 4;             // PL: warp 3 issues
        float acc[DC];
#pragma unroll
        for (int i = 0; i < DC; ++i) acc[i] = 0.f;
        bool ok = true;
        auto drain = [&](int item) -> bool {
            const int b = item & 1;
            if (!mbar_wait_warp(&tfull_bar[b], (item >> 1) & 1, p.wait_ns)) return false;
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * p.ncta);
            if constexpr (PL) {
#pragma unroll
                for (int n0 = 0; n0 < DC; n0 += 16) {
                    if (c0 + n0 < N) {   // N is a multiple of 16
                        uint32_t v[16];
                        tmem_ld16(ta + (uint32_t)(c0 + n0), v);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[n0 + i] += __uint_as_float(v[i]);
                    }
                }
            } else {
#pragma unroll
                for (int n0 = 0; n0 < kTcMaxN; n0 += 32) {
                    if (n0 < N) {
                        uint32_t v[32];
                        tmem_ld32(ta + (uint32_t)n0, v);
                        tmem_wait_ld();
                        // N is a multiple of 16: the upper half of the last load may be past N
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (n0 + i < kTcMaxN && (i < 16 || n0 + 16 < N))
                                acc[n0 + i] += __uint_as_float(v[i]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty_bar[b]);
            return true;
        };
        if (!issuer) {
            for (int item = 0; item < n_items && ok; ++item) ok = drain(item);
        } else {
            // lane 0 issues item i; the whole warp then drains item i - 1 while item i runs
            int seg = 0, chunk = 0;
            while (seg < nseg && !active(seg)) ++seg;
            SegInfo si{};
            if (seg < nseg) si = seg_info(p, t, tt, seg, chunk_elems);
            for (int item = 0; item < n_items && ok; ++item) {
                int good = 1;
                if (lane == 0) {
                    const int stage = item % p.nstages, b = item & 1;
                    if (!mbar_wait(&full_bar[stage], (item / p.nstages) & 1, p.wait_ns) ||
                        !mbar_wait(&bulk_bar[stage], (item / p.nstages) & 1, p.wait_ns) ||
                        (item >= 2 && !mbar_wait(&tempty_bar[b], ((item >> 1) - 1) & 1, p.wait_ns)) ||
                        *(volatile int *)&abort_flag) {
                        good = 0;
                    } else {
                        issue_item(stage, b, si, chunk);
                        if (++chunk == si.nchunks) {
                            chunk = 0;
                            ++seg;
                            while (seg < nseg && !active(seg)) ++seg;
                            if (seg < nseg) si = seg_info(p, t, tt, seg, chunk_elems);
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, good, 0) != 0;
                if (ok && item >= 1) ok = drain(item - 1);
            }
            if (ok && n_items >= 1) ok = drain(n_items - 1);
            // every MMA issued (also before an abort) completes before the tensor memory is freed
            if (lane == 0) {
                mma_commit(&fin_bar);
                if (!mbar_wait(&fin_bar, 0, kWaitNs)) atomicExch(p.err, FMM_ETIMEOUT);
            }
            __syncwarp();
        }
        // epilogue: this thread's row (q * 32 + lane) and columns [c0, c0 + DC)
        const int row = q * 32 + lane;
        const int b = row < t.nrows ? box[row] : -1;
        if (!ok) {
            atomicExch(p.err, FMM_ETIMEOUT);
            *(volatile int *)&abort_flag = 1;
        } else {
            if (b >= 0 && g.Y) {   // FP32 rows (alone, or beside split planes for a later gather)
                float *y = (float *)g.Y + (size_t)b * g.ldy + n_lo;
#pragma unroll
                for (int n0 = 0; n0 < DC; n0 += 4) {
                    const int col = c0 + n0;
                    if (col < N) {
                        float4 o = make_float4(g.alpha * acc[n0], g.alpha * acc[n0 + 1], g.alpha * acc[n0 + 2],
                                               g.alpha * acc[n0 + 3]);
                        if (g.accumulate) {
                            const float4 old = *reinterpret_cast<const float4 *>(y + col);
                            o.x += old.x, o.y += old.y, o.z += old.z, o.w += old.w;
                        }
                        *reinterpret_cast<float4 *>(y + col) = o;
                    }
                }
            }
        }
        if (ok && b >= 0 && p.yp) {
            // split planes for a later tensor-core gather (BF16 hi/lo[/third] or TF32 big/small)
#pragma unroll
            for (int n0 = 0; n0 < DC; n0 += 8) {
                const int col = c0 + n0;
                if (col < N) {
                    const size_t e = (size_t)b * p.yp_ld + n_lo + col;
                    if (!TF32) {
                        uint32_t w[3][4];
#pragma unroll
                        for (int i = 0; i < 8; i += 2) {
                            uint32_t h[2], l[2], m[2];
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                const float x = g.alpha * acc[n0 + i + j];
                                h[j] = bf16_bits(x);
                                const float r1 = x - bf16_val(h[j]);
                                l[j] = bf16_bits(r1);
                                m[j] = bf16_bits(r1 - bf16_val(l[j]));
                            }
                            w[0][i / 2] = h[0] | (h[1] << 16);
                            w[1][i / 2] = l[0] | (l[1] << 16);
                            w[2][i / 2] = m[0] | (m[1] << 16);
                        }
#pragma unroll
                        for (int pl = 0; pl < 3; ++pl)
                            if (pl < p.nplanes)
                                *reinterpret_cast<uint4 *>(p.yp + pl * p.yp_plane + e * 2) =
                                    make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
                    } else {
                        uint32_t bb[8], ss[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float x = g.alpha * acc[n0 + i];
                            bb[i] = tf32_round(x);
                            ss[i] = tf32_round(x - __uint_as_float(bb[i]));
                        }
                        uint4 *d0 = reinterpret_cast<uint4 *>(p.yp + e * 4);
                        uint4 *d1 = reinterpret_cast<uint4 *>(p.yp + p.yp_plane + e * 4);
                        d0[0] = make_uint4(bb[0], bb[1], bb[2], bb[3]);
                        d0[1] = make_uint4(bb[4], bb[5], bb[6], bb[7]);
                        d1[0] = make_uint4(ss[0], ss[1], ss[2], ss[3]);
                        d1[1] = make_uint4(ss[4], ss[5], ss[6], ss[7]);
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

template <bool TF32>
__global__ void __launch_bounds__(kTcThreads, 1) gemm_tc_kernel(const __grid_constant__ TcDev p) {
    tc_body<TF32, false>(p);
}

// Plane layout: capped at 120 registers a thread (46K for the CTA), so that near-field CTAs fit
// beside it on an SM.
template <bool TF32>
__global__ void __maxnreg__(120) gemm_tc_plane_kernel(const __grid_constant__ TcDev p) {
    tc_body<TF32, true>(p);
}

// ---------------------------------------------------------------------------------------
// host side: operand planes and launch
// ---------------------------------------------------------------------------------------
namespace {

// planes of the operands in a precision mode
int planes_of(int prec) { return prec == FMM_BF16X6 ? 3 : 2; }

uint16_t host_bf16(float x) {   // round to nearest even
    uint32_t u;
    std::memcpy(&u, &x, 4);
    uint32_t lsb = (u >> 16) & 1u;
    u += 0x7fffu + lsb;
    return (uint16_t)(u >> 16);
}
float host_bf16_val(uint16_t b) {
    uint32_t u = (uint32_t)b << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}
uint32_t host_tf32(float x) {   // round to nearest (ties away), 10 explicit mantissa bits
    uint32_t u;
    std::memcpy(&u, &x, 4);
    u += 0x1000u;
    return u & 0xffffe000u;
}
float host_f(uint32_t u) {
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}
}  // namespace

// rows x cols FP64 (row-major) -> the split planes of the padded rows_p x cols_p operand, in
// the stage layout [chunk][plane][rows_p x 128 B, SWIZZLE_128B], appended to `out`.
static void tc_pack(int prec, const double *w, int rows, int cols, int rows_p, int cols_p,
                    std::vector<unsigned char> &out) {
    const bool tf32 = prec == FMM_TF32X3;
    const int np = planes_of(prec);
    const int esz = tf32 ? 4 : 2;
    const int ce = kAtomBytes / esz;
    const int nchunks = (cols_p + ce - 1) / ce;
    const size_t plane_bytes = (size_t)rows_p * kAtomBytes;
    const size_t base = out.size();
    out.resize(base + (size_t)nchunks * np * plane_bytes, 0);
    unsigned char *h = out.data() + base;
    for (int r = 0; r < rows; ++r)
        for (int c = 0; c < cols; ++c) {
            const double x = w[(size_t)r * cols + c];
            const int chunk = c / ce, kin = c % ce;
            const int unit = (kin * esz) >> 4, within = (kin * esz) & 15;
            const size_t off = (size_t)(r >> 3) * 1024 + (r & 7) * 128 + ((unit ^ (r & 7)) << 4) + within;
            unsigned char *dst = h + (size_t)chunk * np * plane_bytes + off;
            if (tf32) {
                const uint32_t b = host_tf32((float)x);
                const uint32_t sm = host_tf32((float)(x - (double)host_f(b)));
                std::memcpy(dst, &b, 4);
                std::memcpy(dst + plane_bytes, &sm, 4);
            } else {
                const uint16_t b0 = host_bf16((float)x);
                const double r1 = x - (double)host_bf16_val(b0);
                const uint16_t b1 = host_bf16((float)r1);
                const double r2 = r1 - (double)host_bf16_val(b1);
                const uint16_t b2 = host_bf16((float)r2);
                const uint16_t v[3] = {b0, b1, b2};
                for (int pl = 0; pl < np; ++pl) std::memcpy(dst + pl * plane_bytes, &v[pl], 2);
            }
        }
}

// `count` operators of rows x cols (consecutive in w) packed into one allocation
static cudaError_t tc_upload_many(fmm_ctx *ctx, const double *w, int count, int rows, int cols,
                                  int rows_p, int cols_p, TcMat *out) {
    std::vector<unsigned char> h;
    for (int k = 0; k < count; ++k)
        tc_pack(ctx->opt.precision, w + (size_t)k * rows * cols, rows, cols, rows_p, cols_p, h);
    void *d = nullptr;
    FMM_CUDA_TRY(dev_malloc(&d, h.size()));
    ctx->op_allocs.push_back(d);
    FMM_CUDA_TRY(cudaMemcpy(d, h.data(), h.size(), cudaMemcpyHostToDevice));
    out->planes[0] = d;
    out->rows = rows_p;
    out->cols = cols_p;
    out->nplanes = planes_of(ctx->opt.precision);
    out->bytes = h.size() / count;   // bytes of one operator (the stride)
    return cudaSuccess;
}

static cudaError_t tc_upload_set(fmm_ctx *ctx, const HostOps &h, bool adjoint, const OpSet &o, TcOpSet &t) {
    const int ns = h.ns, nsp = o.nsp;
    const auto &U = adjoint ? h.a_up : h.up;
    const auto &D = adjoint ? h.a_down : h.down;
    std::vector<double> ups;
    for (int c = 0; c < 8; ++c) ups.insert(ups.end(), U[c].begin(), U[c].end());
    FMM_CUDA_TRY(tc_upload_many(ctx, ups.data(), 8, ns, ns, nsp, nsp, &t.up));
    // the 8 D2D operators in one allocation, one view each
    {
        std::vector<double> downs;
        for (int c = 0; c < 8; ++c) downs.insert(downs.end(), D[c].begin(), D[c].end());
        TcMat all;
        FMM_CUDA_TRY(tc_upload_many(ctx, downs.data(), 8, ns, ns, nsp, nsp, &all));
        for (int c = 0; c < 8; ++c) {
            t.down[c] = all;
            t.down[c].planes[0] = (unsigned char *)all.planes[0] + (size_t)c * all.bytes;
        }
    }
    FMM_CUDA_TRY(tc_upload_many(ctx, (adjoint ? h.a_compress : h.compress).data(), 1, o.kin, ns, o.kinp, nsp,
                                &t.compress));
    FMM_CUDA_TRY(tc_upload_many(ctx, (adjoint ? h.a_decompress : h.decompress).data(), 1, ns, o.kout, nsp,
                                o.koutp, &t.decompress));
    FMM_CUDA_TRY(tc_upload_many(ctx, (adjoint ? h.a_stencil : h.stencil).data(), kNumTransfer, o.kout, o.kin,
                                o.koutp, o.kinp, &t.stencil));
    return cudaSuccess;
}

cudaError_t tc_upload_operators(fmm_ctx *ctx) {
    for (int l = 0; l <= kMaxDepth; ++l) {   // each distinct host set once, as the SIMT copies
        int first = -1;
        for (int k = 0; k < l && first < 0; ++k)
            if (ctx->host_ops[k] == ctx->host_ops[l]) first = k;
        if (first >= 0) {
            ctx->tc_fwd[l] = ctx->tc_fwd[first];
            ctx->tc_adj[l] = ctx->tc_adj[first];
            continue;
        }
        ctx->tc_owned.push_back(ctx->tc_fwd[l] = new TcOpSet());
        ctx->tc_owned.push_back(ctx->tc_adj[l] = new TcOpSet());
        FMM_CUDA_TRY(tc_upload_set(ctx, *ctx->host_ops[l], false, ctx->fwd[l], *ctx->tc_fwd[l]));
        FMM_CUDA_TRY(tc_upload_set(ctx, *ctx->host_ops[l], true, ctx->adj[l], *ctx->tc_adj[l]));
    }
    return cudaSuccess;
}

void tc_free(fmm_ctx *ctx) {
    for (TcOpSet *t : ctx->tc_owned) delete t;
    ctx->tc_owned.clear();
    for (int l = 0; l <= kMaxDepth; ++l) ctx->tc_fwd[l] = ctx->tc_adj[l] = nullptr;
}

GemmDev make_gemm_dev(const fmm_ctx *ctx, const GemmCall &c);

cudaError_t gemm_tc(const fmm_ctx *ctx, const GemmCall &c, int op_id, cudaStream_t s) {
    if (c.tiles || c.rows) return cudaErrorNotSupported;   // box subsets: SIMT form only
    const bool adj = op_id >= OP_COUNT;
    const int op = op_id % OP_COUNT;
    // the output level's operators; PARENT2's D2D segment those of the parent level
    const TcOpSet &T = adj ? *ctx->tc_adj[c.level] : *ctx->tc_fwd[c.level];
    const int lp = c.level > 0 ? c.level - 1 : 0;
    const TcOpSet &T1 = adj ? *ctx->tc_adj[lp] : *ctx->tc_fwd[lp];
    TcDev p{};
    p.g = make_gemm_dev(ctx, c);
    const TileSet &ts = (c.mode == GM_STENCIL || c.mode == GM_PARENT2) ? ctx->tiles_cls[c.level]
                                                                       : ctx->tiles_plain[c.level];
    if (ts.ntiles == 0) return cudaSuccess;
    p.g.tiles = ts.tiles;
    p.g.masks = ts.masks;
    if (c.mode == GM_STENCIL && ctx->masks_ev) FMM_CUDA_TRY(cudaStreamWaitEvent(s, ctx->masks_ev, 0));
    switch (op) {
        case OP_UP: p.Wt0 = (const unsigned char *)T.up.planes[0]; p.wt_stride = (long long)T.up.bytes; break;
        case OP_COMPRESS: p.Wt0 = (const unsigned char *)T.compress.planes[0]; break;
        case OP_STENCIL: p.Wt0 = (const unsigned char *)T.stencil.planes[0]; p.wt_stride = (long long)T.stencil.bytes; break;
        case OP_DECOMPRESS:
            p.Wt0 = (const unsigned char *)T.decompress.planes[0];
            for (int k = 0; k < 8; ++k) p.Wt1[k] = (const unsigned char *)T1.down[k].planes[0];
            break;
        default: return cudaErrorInvalidValue;
    }
    const int prec = ctx->opt.precision;
    p.tf32 = prec == FMM_TF32X3;
    p.nplanes = planes_of(prec);
    if (p.nplanes == 3) {
        const int a[6] = {2, 1, 0, 1, 0, 0}, b[6] = {0, 1, 2, 0, 1, 0};
        p.nprod = 6;
        for (int i = 0; i < 6; ++i) p.prod_a[i] = a[i], p.prod_b[i] = b[i];
    } else {
        const int a[3] = {1, 0, 0}, b[3] = {0, 1, 0};
        p.nprod = 3;
        for (int i = 0; i < 3; ++i) p.prod_a[i] = a[i], p.prod_b[i] = b[i];
    }
    if (c.n_out % 16 != 0 || (c.k0 % 16) != 0 || (c.X1 && c.k1 % 16 != 0)) return cudaErrorInvalidValue;
    const int nsplit = (c.n_out + kTcMaxN - 1) / kTcMaxN;
    p.ncta = round_up((c.n_out + nsplit - 1) / nsplit, 16);
    const int stage_bytes = p.nplanes * (kTcRows + p.ncta) * kAtomBytes;
    // 227 KB per CTA in all: the stages, 1 KB of alignment slack and the static shared memory.
    // The plane layout keeps two stages, which leaves room on the SM for near-field CTAs.
    const bool plane = c.Xp != nullptr;
    auto kern = plane ? (p.tf32 ? gemm_tc_plane_kernel<true> : gemm_tc_plane_kernel<false>)
                      : (p.tf32 ? gemm_tc_kernel<true> : gemm_tc_kernel<false>);
    const int threads = plane ? 384 : kTcThreads;
    int most = 0;
    FMM_CUDA_TRY(allow_all_shared(kern, &most));
    p.nstages = std::min(plane ? kPlaneStages : 4, (most - 1024) / stage_bytes);
    if (p.nstages < 2) return cudaErrorInvalidValue;
    // two accumulators of ncta columns; the drain reads 32 columns at a time, so the last read
    // of the second accumulator may extend 16 columns past it: keep that inside the allocation
    int cols = 32;
    while (cols < 2 * p.ncta + 16) cols <<= 1;
    if (cols > 512) return cudaErrorInvalidValue;
    p.tmem_cols = cols;
    p.err = ctx->dev_flag;
    p.wait_ns = ctx->tc_wait_ns;
    if (c.Xp) {
        // A rows from split planes: K of the segment must be the planes' width
        if (c.mode == GM_PARENT2) return cudaErrorInvalidValue;
        if (((uintptr_t)c.Xp & 15) || ((c.xp_ld * (p.tf32 ? 4 : 2)) & 15) || (c.xp_plane & 15))
            return cudaErrorInvalidValue;
        p.a_planes = 1;
        p.xp = (const unsigned char *)c.Xp;
        p.xp_plane = c.xp_plane;
        p.xp_ld = c.xp_ld;
    }
    if (c.Yp) {
        p.yp = (unsigned char *)c.Yp;
        p.yp_plane = c.yp_plane;
        p.yp_ld = c.yp_ld;
    }
    const size_t smem = (size_t)p.nstages * stage_bytes + 1024;
    kern<<<dim3(ts.ntiles, (c.n_out + p.ncta - 1) / p.ncta), threads, smem, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

}  // namespace fmm
