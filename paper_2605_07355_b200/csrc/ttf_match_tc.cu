// Pointwise Matching with Local Window Search and Threshold Gating (Eqs. pi, argmax, dst, gating, mask) for bf16
// clips on the fifth-generation tensor cores: TMA tensor tiles -> shared memory -> tcgen05.mma -> tensor memory.
//
// All tokens of a grid cell share their candidate set, and neighbouring cells share most of it, so the unit of
// work is a TILE of 128 source rows = FR frames x WY grid rows x 4 cells (FR = 32 / WY, WY = 1, 2 or 4), against the
// (WY+2r) x (4+2r) anchor cells around them: one dense contraction
//     D[128 x NB] = A[128 x C] . B[NB x C]^T,     NB = 16 / 32 / 48 >= (WY+2r)(4+2r),
// of which every source row uses its own (2r+1)^2 columns.  Operand traffic is (128 + 18) / 128 = 1.14 x |X| for 32 frames at
// r = 1 instead of 41 / 32 when every cell fetches its own 9 candidates.  Frames that a clip does not have are rows of zeros:
// they cost no traffic, but the stages, norms and epilogue of a whole tile, so clips of few frames take tiles of fewer frames
// and more grid rows (tile_rows; against 32 frames throughout, us per pass: 8 clips of 8 x 32 x 32 x 1024 128 -> 76, 16 of
// 8 x 16 x 16 x 1024 71 -> 46, 7 of 6 x 12 x 7 x 1944 25.4 -> 16.9, 6 of 48 x 14 x 14 x 1024 71.9 -> 64.6, one of
// 9 x 16 x 16 x 4096 26.4 -> 22.8, of 5 x 29 x 13 x 1016 at r = 2 20.2 -> 18.4).
//
//   A tile:  box (64 channels, 4 cells, WY rows, FR frames) of X viewed as [F, H, W, C]; row m = (frame, cell row, cell).
//   B tile:  box (64 channels, 4 + 2r cells, WY + 2r rows, 1 frame) at frame a*, starting r cells up and left of the
//            tile; cells outside the grid arrive as zeros and are left out of the arg max (window clipped to the
//            grid, Eq. pi, with the duplicates of the clipping masked).
//   Both arrive with the 128-byte swizzle, which is the K-major operand layout of tcgen05.mma; a pipeline stage is
//   64 channels (4 MMAs of K = 16).  fp32 accumulation in tensor memory; bf16 products are exact in fp32.
//
// The channel range of a tile is cut into `chunks` consecutive parts, each with an accumulator of its own in tensor
// memory, and a tile is worked on by `pieces` CTAs (a divisor of `chunks`), which take chunks / pieces of the parts each.
// The sums of the parts are added as a binary tree over the parts, so the result depends on `chunks` alone: a clip gives
// the same bits whether it has the GPU to itself (pieces = chunks, so that a small clip still gives about two CTAs per
// SM) or shares a launch with others (fewer pieces, no exchange between CTAs).
// The CTAs of a tile form a thread-block cluster, and each rank finishes 128 / pieces of the rows: when its accumulators
// are complete a rank writes its partial sums of every rank's rows into that rank's shared memory (a region of its own
// beside the ring, so that nobody has to wait for the others' pipelines to drain first) and one cluster barrier follows.
// What comes after the main loop is a serial chain that nothing overlaps, so with several ranks every step of it is spread
// over all 128 epilogue threads: (element, rank) sums, then the norms, then one row per thread.
// Token norms are taken from the tiles themselves: while the pipeline runs, every epilogue thread adds up the squares
// of "its" source row (and the first NCAND threads those of a candidate row) as the stages pass through shared memory.
// Warp roles: 0 TMA producer, 1 tensor-memory owner and MMA issuer, 2-5 epilogue (one tensor-memory lane = one
// source row per thread).
//
// Every mbarrier wait is bounded; a wait that runs out sets the error word of the call, the CTA stops feeding its
// pipeline, waits (bounded again) for the copies it has in flight, frees its tensor memory and returns.
#include <cuda.h>

#include "ttf_internal.cuh"
#include "ttf_async.cuh"
#include "ttf_cluster.cuh"
#include "ttf_tensormap.cuh"

#include <atomic>
#include <mutex>

namespace ttf {

constexpr int kTcWB = 4;                 // cells per strip
constexpr int kTcM = 128;                // source rows of a tile = tensor-memory lanes
constexpr int kTcKC = 64;                // channels per stage (128 bytes: one swizzle row)
constexpr int kTcABytes = kTcM * 128;    // 16 KB
constexpr int kTcThreads = 192;

// ---- PTX wrappers -----------------------------------------------------------------------------------------
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// whole warp: allocates `cols` (a power of two >= 32) columns of tensor memory, base address -> *dst_smem
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[tmem] (+)= A[smem desc] . B[smem desc]^T, issued by one thread
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}
// the barrier receives one arrival when every MMA issued so far by this thread has completed
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 8 NG consecutive fp32 columns of this thread's tensor-memory lane
template <int NG> __device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[NG][8]) {
#pragma unroll
    for (int g = 0; g < NG; ++g)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[g][0]), "=r"(r[g][1]), "=r"(r[g][2]), "=r"(r[g][3]), "=r"(r[g][4]), "=r"(r[g][5]),
                       "=r"(r[g][6]), "=r"(r[g][7])
                     : "r"(taddr + (uint32_t)(g * 8))
                     : "memory");
#pragma unroll
    for (int g = 0; g < NG; ++g)                           // (the registers are operands of the wait, so that nothing that
        asm volatile("tcgen05.wait::ld.sync.aligned;"      // reads them can be moved before it)
                     : "+r"(r[g][0]), "+r"(r[g][1]), "+r"(r[g][2]), "+r"(r[g][3]), "+r"(r[g][4]), "+r"(r[g][5]),
                       "+r"(r[g][6]), "+r"(r[g][7])
                     :: "memory");
}
template <int NG> __device__ __forceinline__ void tmem_add(uint32_t (&a)[NG][8], const uint32_t (&b)[NG][8]) {
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int e = 0; e < 8; ++e) a[g][e] = __float_as_uint(__uint_as_float(a[g][e]) + __uint_as_float(b[g][e]));
}
__device__ __forceinline__ void epilogue_bar_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// K-major operand tile with the 128-byte swizzle: rows of 128 bytes, groups of 8 rows 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);          // start address, 16-byte units
    d |= (uint64_t)1 << 16;                               // leading byte offset (not used by swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                     // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                               // descriptor version of sm_100
    d |= (uint64_t)2 << 61;                               // 128-byte swizzle
    return d;
}
// bf16 x bf16 -> fp32, A and B K-major, M = 128, N = NB
__host__ __device__ constexpr uint32_t idesc_bf16(int NB) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
}

// ---- the kernel -------------------------------------------------------------------------------------------
// MMA N of a tile of `wy` grid rows
constexpr int tile_columns(int r, int wy) { return ((kTcWB + 2 * r) * (wy + 2 * r) + 15) / 16 * 16; }
// Chunks of a tile at most: the same whatever its rows, so that no sum in tensor memory has more terms than in tiles of one row
// (a tensor-memory accumulator truncates: similarities of 8 x 8 x 8 x 4096 at r = 1 against 64 bits 5.4e-7 with eight chunks,
// 1.3e-6 with four, which took 20.5 us per pass against 17.3; 4 x 12 x 12 x 4096 1.1e-6 -> 4.9e-7 and 20.1 -> 17.1 us).
constexpr int max_chunks(int r) { return r == 2 ? 4 : 8; }
// ... and of one CTA (256 columns of tensor memory at most: two CTAs per SM)
constexpr int own_chunks(int nb) { return nb > 32 ? 4 : 8; }

template <int R, int WY> struct TcShape {
    static constexpr int FR = kTcM / (kTcWB * WY);        // frames per tile
    static constexpr int SIDE = 2 * R + 1;
    static constexpr int BW = kTcWB + 2 * R, BH = WY + 2 * R;      // candidate cells: columns, rows
    static constexpr int NCAND = BW * BH;                 // rows the B box delivers
    static constexpr int NB = tile_columns(R, WY);        // MMA N
    static constexpr int BBYTES = NB * 128;
    static constexpr int BBOX = NCAND * 128;              // bytes one B box copy delivers
    static constexpr int STAGE = kTcABytes + BBYTES;
    static constexpr int STAGES = 4;                      // two CTAs per SM with room left for CTAs of other kernels
    static constexpr int WIN = SIDE * SIDE;               // candidates of one source row
    static constexpr int MAXCH = max_chunks(R), OWNCH = own_chunks(NB);
    // what one rank sends another (and itself): window sums and squared norms of the rows the other one finishes,
    // squared norms of the candidates
    static constexpr int XBYTES = (kTcM * (WIN + 1) + MAXCH * NCAND) * 4;                 // received by one rank
    static constexpr int RING = STAGES * STAGE;
    static constexpr int NP = NCAND * 8;                  // (candidate row, 16-byte piece column) pairs
    static constexpr int NORMBYTES = OWNCH * (kTcM + NP) * 4;
};

// m is all ones or zero: a or b without a branch.  (The window of a row starts at one of four columns; as conditional
// expressions the choice became divergent branches, 1400 cycles per row at r = 1 against 110 for the loads from tensor
// memory; 16 logic operations now.)
__device__ __forceinline__ uint32_t pick(uint32_t m, uint32_t a, uint32_t b) { return (a & m) | (b & ~m); }
// binary tree over n = 1, 2, 4 or 8 terms
template <typename Fn> __device__ __forceinline__ float tree_sum(int n, Fn&& term) {
    float v = term(0);
    if (n > 1) v += term(1);
    if (n > 2) v += term(2) + term(3);
    if (n > 4) v += (term(4) + term(5)) + (term(6) + term(7));
    return v;
}

// sum of squares of the 8 bf16 values of a 16-byte piece
__device__ __forceinline__ float ssq8(const uint4& v, float acc) {
    float x;
    x = bf16_lo(v.x); acc = fmaf(x, x, acc); x = bf16_hi(v.x); acc = fmaf(x, x, acc);
    x = bf16_lo(v.y); acc = fmaf(x, x, acc); x = bf16_hi(v.y); acc = fmaf(x, x, acc);
    x = bf16_lo(v.z); acc = fmaf(x, x, acc); x = bf16_hi(v.z); acc = fmaf(x, x, acc);
    x = bf16_lo(v.w); acc = fmaf(x, x, acc); x = bf16_hi(v.w); acc = fmaf(x, x, acc);
    return acc;
}

template <int R, int WY, int G>
__global__ void __launch_bounds__(kTcThreads)
k_match_tc(const __grid_constant__ ClipMaps<G> maps, int F, int H, int W, int C, float t, AnchorSrc asrc, int lpieces, int lchunks,
           float* __restrict__ shat, int* __restrict__ dst, unsigned char* __restrict__ keep, int* __restrict__ cnt,
           int wait_limit, int tx_extra, int stream_once, size_t sstride, int* fuse_cnt)
{
    using S = TcShape<R, WY>;
    const bool backwards = gridDim.y == 1 || stream_once;
    const unsigned clip = backwards ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
    const CUtensorMap& mapA = maps.a[clip];
    const CUtensorMap& mapB = maps.b[clip];
    asrc = clip_block(asrc, sstride, clip); cnt = clip_block(cnt, sstride, clip);
    shat = clip_block(shat, sstride, clip); dst = clip_block(dst, sstride, clip); keep = clip_block(keep, sstride, clip);
    extern __shared__ unsigned char dyn_raw[];
    __shared__ uint64_t bar_full[S::STAGES], bar_empty[S::STAGES], bar_acc;
    __shared__ uint32_t s_tmem;
    __shared__ int s_err;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = H * W;
    const int xs_n = (W + kTcWB - 1) / kTcWB;
    // A launch over one clip walks its tiles backwards: the sweep has gone forwards, so what it read last is still in L2,
    // and the gather, which goes forwards again, finds what is matched last.  (64 x 16 x 16 x 4096: 81.9 -> 79.0 us per
    // pass, 64 x 32 x 32 x 4096 with r = 2: 255.5 -> 252.1.)  Over several clips it needs the L2 hints of stream_once as well.
    const unsigned walk = backwards ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int pieces = 1 << lpieces;
    const int tile = (int)(walk >> lpieces);
    const int piece = pieces > 1 ? (int)cluster_rank() : 0;        // = blockIdx.x % pieces
    const int ys_n = (H + WY - 1) / WY;
    const int kg = tile / (ys_n * xs_n), rem = tile - kg * (ys_n * xs_n);
    const int y0 = rem / xs_n * WY, x0 = rem % xs_n * kTcWB;
    const int k0 = kg * S::FR;
    const int nst_all = (C + kTcKC - 1) / kTcKC;
    const int nch = 1 << (lchunks - lpieces);              // this CTA's chunks: ch0 .. ch0 + nch - 1
    const int ch0 = piece * nch;
    auto chunk_begin = [&](int c) { return (nst_all * c) >> lchunks; };
    const int st0 = chunk_begin(ch0), nst = chunk_begin(ch0 + nch) - st0;
    uint32_t tmem_cols = 32;
    while (tmem_cols < (uint32_t)(nch * S::NB)) tmem_cols *= 2;

    // 1024-byte aligned stage ring (the swizzle pattern is a function of the shared-memory address)
    const uint32_t dyn_base = (smem_u32(dyn_raw) + 1023u) & ~1023u;
    unsigned char* dyn = dyn_raw + (dyn_base - smem_u32(dyn_raw));

    trace_mark(asrc.hdr, 2, false);
    if (tid == 0) {
        // a stage is full when its two copies have landed, and free again when the MMAs that read it have completed
        // and each of the four epilogue warps has taken its share of the norms from it
        for (int s = 0; s < S::STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 5); }
        mbar_init(&bar_acc, 1);
        mbar_init_fence();
        s_err = 0;
        tensormap_prefetch(&mapA);
        tensormap_prefetch(&mapB);
    }
    // the B rows beyond the box (NCAND .. NB-1) are never written by a copy: zero them once
    constexpr int PAD = (S::BBYTES - S::BBOX) / 16;        // 16-byte pieces per stage
    for (int i = tid; i < S::STAGES * PAD; i += kTcThreads) {
        const int s = i / (PAD > 0 ? PAD : 1), o = i - s * PAD;
        reinterpret_cast<uint4*>(dyn + (size_t)s * S::STAGE + kTcABytes + S::BBOX)[o] = make_uint4(0, 0, 0, 0);
    }
    fence_async_smem();
    if (warp == 1) tmem_alloc(&s_tmem, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    if (pieces > 1) { cluster_arrive(); cluster_wait(); }  // every CTA of the tile is running: remote writes may come

    // everything upstream (the anchor, and whatever produced X) is complete after this wait
    trace_mark(asrc.hdr, 11, false); trace_mark(asrc.hdr, 11, true);     // set-up done
    pdl_wait();
    trace_mark(asrc.hdr, 5, false);
    const int a = asrc.fixed >= 0 ? asrc.fixed : __ldcg(asrc.hdr + HDR_ANCHOR);
    if (blockIdx.x == 0 && tid == 0 && asrc.fixed >= 0) {
        if (asrc.begins) clear_words(asrc.hdr, false);
        asrc.hdr[HDR_ANCHOR] = a;                // the gather reads it from here
        if (asrc.out_anchor) *asrc.out_anchor = a;
    }

    // epilogue-thread state that outlives the role code
    const int q = warp & 3;                                // tensor-memory lane quadrant an epilogue warp may read
    const int m = q * 32 + lane;                           // source row of an epilogue thread: (frame, cell row, cell column)
    const int et = (warp - 2) * 32 + lane;                 // 0..127 among the epilogue threads
    float* const s_na = reinterpret_cast<float*>(dyn + S::RING + S::XBYTES);      // [chunk][row] squared norms
    float* const s_nbp = s_na + S::OWNCH * kTcM;           // [chunk][candidate row, piece column]
    const int dx = m & 3, dy = (m >> 2) & (WY - 1);
    float win[S::WIN];                                     // this row's window of dot products
    float na = 0.f, nb = 0.f;                              // squared norm of source row m / of candidate row et

    if (warp == 0) {
        // ---- producer: one lane issues the tile copies of every stage ----------------------------------------
        if (lane == 0) {
            int issued = 0;
            const uint64_t once = l2_evict_first_policy();
            for (int it = 0; it < nst; ++it) {
                const int s = it % S::STAGES;
                if (it >= S::STAGES && !mbar_wait(&bar_empty[s], ((it / S::STAGES) & 1) ^ 1, wait_limit)) { atomicExch(&s_err, 1); break; }
                if (*(volatile int*)&s_err) break;
                unsigned char* sa = dyn + (size_t)s * S::STAGE;
                const int c0 = (st0 + it) * kTcKC;
                mbar_arrive_expect_tx(&bar_full[s], kTcABytes + S::BBOX + (uint32_t)tx_extra);   // (extra: test hook only)
                // source rows are read by this tile alone: in a schedule that streams the next clip into L2 meanwhile,
                // their lines are the ones to give up first (the candidate rows are shared with neighbouring tiles)
                if (stream_once) tma_load_4d_hint(sa, &mapA, c0, x0, y0, k0, &bar_full[s], once);
                else tma_load_4d(sa, &mapA, c0, x0, y0, k0, &bar_full[s]);
                tma_load_4d(sa + kTcABytes, &mapB, c0, x0 - R, y0 - R, a, &bar_full[s]);
                issued = it + 1;
            }
            trace_mark_any(asrc.hdr, 12, false); trace_mark_any(asrc.hdr, 12, true);   // all copies issued
            if (*(volatile int*)&s_err) {
                // copies already issued still land in this CTA's shared memory: wait (bounded) for the stages that
                // nobody consumed before the CTA is allowed to exit
                for (int it = issued > S::STAGES ? issued - S::STAGES : 0; it < issued; ++it)
                    mbar_wait(&bar_full[it % S::STAGES], (it / S::STAGES) & 1, wait_limit);
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer: one lane, four K = 16 steps per stage -----------------------------------------------
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(S::NB);
            int ch = 0, begin = 0, end = chunk_begin(ch0 + 1) - st0;     // stages of the chunk
            for (int it = 0; it < nst; ++it) {
                const int s = it % S::STAGES;
                if (it == end) { ++ch; begin = end; end = chunk_begin(ch0 + ch + 1) - st0; }
                if (!mbar_wait(&bar_full[s], (it / S::STAGES) & 1, wait_limit)) { atomicExch(&s_err, 1); break; }
                tc_fence_after();
                const uint32_t sa = dyn_base + (uint32_t)s * S::STAGE;
                const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + kTcABytes);
#pragma unroll
                for (int k = 0; k < kTcKC / 16; ++k)       // 32 bytes further along K inside the swizzle row
                    umma_bf16(tmem + (uint32_t)(ch * S::NB), da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc,
                              it > begin || k > 0);
                umma_commit(&bar_empty[s]);                // one of the five arrivals that free the stage
            }
            umma_commit(&bar_acc);                         // accumulator complete (also arrives after a give-up)
        }
    } else {
        // ---- epilogue warps, part 1: while the pipeline runs, the squared norms of the rows that pass through
        // shared memory (source row m by every thread, candidate row et by the first NCAND threads).  A row is 128
        // bytes per stage; its 16-byte pieces sit at (piece ^ (row & 7)) (the 128-byte swizzle), and a sum of
        // squares does not care in which order it meets them ---------------------------------------------------
        bool ok = true;
        constexpr int NP = S::NP;
        constexpr int PP = (NP + 127) / 128;               // pairs per epilogue thread
        float na8[8], nbq[PP];                             // one running sum per piece column: eight short chains
#pragma unroll
        for (int c = 0; c < 8; ++c) na8[c] = 0.f;
#pragma unroll
        for (int u = 0; u < PP; ++u) nbq[u] = 0.f;
        int ch = 0, end = chunk_begin(ch0 + 1) - st0;
        for (int it = 0; it < nst; ++it) {
            const int s = it % S::STAGES;
            if (!mbar_wait(&bar_full[s], (it / S::STAGES) & 1, wait_limit)) { atomicExch(&s_err, 1); ok = false; break; }
            const unsigned char* sa = dyn + (size_t)s * S::STAGE;
            const uint4* rowa = reinterpret_cast<const uint4*>(sa + (size_t)m * 128);
            uint4 va[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) va[c] = rowa[c ^ (m & 7)];
            uint4 vb[PP];
#pragma unroll
            for (int u = 0; u < PP; ++u) {
                const int pr = et + u * 128, row = pr >> 3, pc = pr & 7;
                vb[u] = pr < NP ? reinterpret_cast<const uint4*>(sa + kTcABytes + (size_t)row * 128)[pc ^ (row & 7)]
                                : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) na8[c] = ssq8(va[c], na8[c]);
#pragma unroll
            for (int u = 0; u < PP; ++u) nbq[u] = ssq8(vb[u], nbq[u]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_empty[s]);
            if (it + 1 == end) {                           // a chunk is complete: put its norms away
                s_na[ch * kTcM + m] = ((na8[0] + na8[1]) + (na8[2] + na8[3])) + ((na8[4] + na8[5]) + (na8[6] + na8[7]));
#pragma unroll
                for (int c = 0; c < 8; ++c) na8[c] = 0.f;
#pragma unroll
                for (int u = 0; u < PP; ++u) {
                    if (et + u * 128 < NP) s_nbp[ch * NP + et + u * 128] = nbq[u];
                    nbq[u] = 0.f;
                }
                ++ch;
                end = chunk_begin(ch0 + ch + 1) - st0;
            }
        }
        if (et == 0) { trace_mark_any(asrc.hdr, 13, false); trace_mark_any(asrc.hdr, 13, true); }   // norms done
        // ---- part 2: the accumulators, added up over this CTA's chunks ---------------------------------------------
        if (ok) ok = mbar_wait(&bar_acc, 0, wait_limit);
        if (!ok) atomicExch(&s_err, 1);                    // (what follows then works on whatever is there: the call has failed)
        if (et == 0) { trace_mark_any(asrc.hdr, 14, false); trace_mark_any(asrc.hdr, 14, true); }   // accumulator complete
        tc_fence_after();
        // The gather may be scheduled from here on.  (Not earlier: its CTAs would take the places of other kernels' CTAs and
        // sit out the main loop; 24 x 24 x 24 x 2048: 45.8 us per pass with the trigger at the start, 42.3 here.)
        pdl_launch_dependents();
        epilogue_bar_sync();                               // the norms of the chunks are visible
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        constexpr int NG = (S::NCAND + 7) / 8;
        uint32_t d[NG][8];
        tmem_ld<NG>(lanes, d);
        if (nch > 1) {
            uint32_t x[NG][8], z[NG][8];
            tmem_ld<NG>(lanes + (uint32_t)S::NB, x);
            tmem_add<NG>(d, x);
#pragma unroll 1
            for (int h = 2; h < nch; h += 2) {             // nch = 4 or 8: pairs (2,3) | ((4,5), (6,7))
                tmem_ld<NG>(lanes + (uint32_t)(h * S::NB), x);
                tmem_ld<NG>(lanes + (uint32_t)((h + 1) * S::NB), z);
                tmem_add<NG>(x, z);
                if (S::OWNCH > 4 && h == 4) {
                    uint32_t u[NG][8];
                    tmem_ld<NG>(lanes + (uint32_t)(6 * S::NB), u);
                    tmem_ld<NG>(lanes + (uint32_t)(7 * S::NB), z);
                    tmem_add<NG>(u, z);
                    tmem_add<NG>(x, u);
                    h = 6;
                }
                tmem_add<NG>(d, x);
            }
        }
        // this row's window: candidate (wy, wx) is column (dy + wy) * BW + dx + wx of the tile
        const uint32_t by1 = (dx & 1) ? 0xffffffffu : 0u, by2 = (dx & 2) ? 0xffffffffu : 0u;
        const uint32_t dy1 = (dy & 1) ? 0xffffffffu : 0u, dy2 = (dy & 2) ? 0xffffffffu : 0u;
        auto col = [&](int yy, int n) { return d[(yy * S::BW + n) / 8][(yy * S::BW + n) % 8]; };
        auto col2 = [&](int yy, int n) { return WY > 2 ? pick(dy2, col(yy + (WY > 2 ? 2 : 0), n), col(yy, n)) : col(yy, n); };
        auto row_col = [&](int yy, int n) { return WY > 1 ? pick(dy1, col2(yy + (WY > 1 ? 1 : 0), n), col2(yy, n)) : col2(yy, n); };
#pragma unroll
        for (int wy = 0; wy < S::SIDE; ++wy) {
            uint32_t c[S::BW], e[S::SIDE + 2];
#pragma unroll
            for (int n = 0; n < S::BW; ++n) c[n] = row_col(wy, n);
#pragma unroll
            for (int n = 0; n < S::SIDE + 2; ++n) e[n] = pick(by1, c[n + 1], c[n]);
#pragma unroll
            for (int wx = 0; wx < S::SIDE; ++wx) win[wy * S::SIDE + wx] = __uint_as_float(pick(by2, e[wx + 2], e[wx]));
        }
        na = tree_sum(nch, [&](int c) { return s_na[c * kTcM + m]; });
        if (et < S::NCAND)
            nb = tree_sum(nch, [&](int c) {
                const float* pp = s_nbp + c * NP + et * 8;
                return ((pp[0] + pp[1]) + (pp[2] + pp[3])) + ((pp[4] + pp[5]) + (pp[6] + pp[7]));
            });
    }

    const int per = kTcM >> lpieces;                       // rank p of the cluster finishes rows [p * per, (p + 1) * per)
    const int rows_end = per * (S::WIN + 1);               // a share: [window sum 0 .. WIN-1, norm][row], candidate norms
    const int seg = rows_end + S::NCAND;
    float* const x_in = reinterpret_cast<float*>(dyn + S::RING);         // [rank][seg]
    if (pieces > 1) {
        if (warp >= 2) {
            const int owner = m >> (7 - lpieces);
            const uint32_t own_share = dyn_base + S::RING + (uint32_t)(piece * seg) * 4;
            uint32_t to = cluster_addr(own_share + (uint32_t)(m & (per - 1)) * 4, (uint32_t)owner);
#pragma unroll
            for (int c = 0; c < S::WIN; ++c, to += (uint32_t)per * 4) st_cluster_f32(to, win[c]);
            st_cluster_f32(to, na);
            if (et < S::NCAND)
                for (int p = 0; p < pieces; ++p)
                    st_cluster_f32(cluster_addr(own_share + (uint32_t)(rows_end + et) * 4, (uint32_t)p), nb);
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    }

    if (warp >= 2) {
        // ---- epilogue, part 3 (the rows this rank finishes): cosine, arg max over the window clipped to the grid, gate --
        float* const s_rb = x_in + rows_end;               // 1 / max(||x||, floor) of the candidates
        int row = m;
        if (pieces > 1) {
            for (int e = et; e < seg; e += 128) {          // (an element is read and overwritten by the same thread)
                float v = tree_sum(pieces, [&](int p) { return x_in[p * seg + e]; });
                if (e >= rows_end - per) v = 1.0f / fmaxf(sqrtf(v), kNormFloor);     // ... and of the rows
                x_in[e] = v;
            }
            epilogue_bar_sync();
            row = piece * per + et;
            if (et < per) {
#pragma unroll
                for (int c = 0; c < S::WIN; ++c) win[c] = x_in[c * per + et];
                na = x_in[S::WIN * per + et];
            }
        } else {
            if (et < S::NCAND) s_rb[et] = 1.0f / fmaxf(sqrtf(nb), kNormFloor);
            na = 1.0f / fmaxf(sqrtf(na), kNormFloor);
            epilogue_bar_sync();
        }
        const int k = k0 + row / (kTcWB * WY), cell = row & 3, cy = (row >> 2) & (WY - 1), x = x0 + cell, y = y0 + cy;
        const bool mine = pieces > 1 ? et < per : true;
        if (mine && k < F && x < W && y < H && in_bounds(asrc.hdr, 3, (long long)k * N + (long long)y * W + x, (long long)F * N)) {
            const size_t f = (size_t)k * N + (size_t)y * W + x;
            if (k == a) {                                  // anchor tokens are always retained (Eq. mask)
                shat[f] = 1.0f; dst[f] = y * W + x; keep[f] = 1;
            } else {
                float best = -INFINITY;
                int best_j = -1;
#pragma unroll
                for (int wy = 0; wy < S::SIDE; ++wy)       // ascending anchor index among in-grid cells
#pragma unroll
                    for (int wx = 0; wx < S::SIDE; ++wx) {
                        const int yy = y + wy - R, xx = x + wx - R;
                        const float sim = win[wy * S::SIDE + wx] * na * s_rb[(cy + wy) * S::BW + cell + wx];
                        const bool take = ((unsigned)yy < (unsigned)H) & ((unsigned)xx < (unsigned)W) & ((sim > best) | (best_j < 0));
                        best = take ? sim : best;
                        best_j = take ? yy * W + xx : best_j;
                    }
                gate_token(best, best_j, t, f, shat, dst, keep, cnt + k, fuse_cnt);
            }
        }
    }

    // ---- teardown: every role is done with tensor memory before its owner frees it --------------------------
    tc_fence_before();
    __syncthreads();
    trace_mark(asrc.hdr, 2, true);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, tmem_cols);
    }
    if (tid == 0 && s_err) report_give_up(asrc.hdr, asrc.begins);
}

// ---- host side: tensor maps and launch ------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static std::mutex mu;
    static EncodeTiledFn fn = nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

bool make_tensor_map(CUtensorMap* m, const void* X, int dtype, int F, int H, int W, int C, int kc, int bw, int bh, int bf,
                     bool swizzle128) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t es = dtype == 0 ? 4 : 2;
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)F};
    const cuuint64_t strides[3] = {(cuuint64_t)C * es, (cuuint64_t)W * C * es, (cuuint64_t)H * W * C * es};
    const cuuint32_t box[4] = {(cuuint32_t)kc, (cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)bf};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, dtype == 0 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(X),
               dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
               // (256-byte L2 promotion: the next stage reads the next bytes of the same rows; 5 - 9 % faster than 128
               // for the tcgen05 kernel)
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tc_match_eligible(const Problem& p) {
    if (p.dtype != 1 || !p.vec || p.r > 2 || p.C < kTcKC) return false;
    return (long long)tc_match_tiles(p) * 8 < (1LL << 31);
}

static size_t tiles_of(const Problem& p, int wy) {
    const int fr = kTcM / (kTcWB * wy);
    return (size_t)((p.F + fr - 1) / fr) * ((p.H + wy - 1) / wy) * ((p.W + kTcWB - 1) / kTcWB);
}
static int rows_per_stage(const Problem& p, int wy) { return kTcM + (kTcWB + 2 * p.r) * (wy + 2 * p.r); }
static int most_rows(const Problem& p) { return p.r == 2 ? 2 : 4; }       // (r = 2 with four rows would need 64 columns of 128 registers)
// The tile (1, 2 or 4 grid rows, hence 32, 16 or 8 frames) with the fewest rows to fetch, padding and candidates included.
static int fewest_rows(const Problem& p) {
    int best = 1;
    for (int wy = 2; wy <= most_rows(p); wy *= 2)
        if (tiles_of(p, wy) * rows_per_stage(p, wy) < tiles_of(p, best) * rows_per_stage(p, best)) best = wy;
    return best;
}
size_t tc_match_tiles(const Problem& p) { return tiles_of(p, fewest_rows(p)); }

// Parts of a tile's channel range: the largest power of two with which a launch over one clip still fits the GPU in one
// wave of two CTAs per SM, at most max_chunks and at least 2 stages each (4 stages: 16 x 8 x 8 x 512 13.9 us per pass,
// 2: 12.9, 1: 13.3; 16 x 14 x 14 x 512 16.7 / 15.3 / 15.3).  (One CTA per SM with a ring twice as deep measured the same
// alone, 18.8 against 19.2 us on a cold 8B-shaped clip, and slower with other clips' kernels beside it, 34.0 against
// 32.2 us per clip.)
static int split_of(const Problem& p, long long tiles, int most, int sms) {
    const int nst = (p.C + kTcKC - 1) / kTcKC;
    int n = 1;
    while (n * 2 <= most && tiles * (n * 2) <= 2LL * sms && nst / (n * 2) >= 2) n *= 2;
    return n;
}


// How many clusters of n CTAs run at the same time on the current device (asked once).  Two CTAs fit an SM, but the places of a
// cluster lie in one GPC: 148 SMs hold 148 clusters of two, 71 of four, 33 of eight.  (The runtime is asked about a kernel of
// the same shape that uses no tensor memory: for one that does it counts one CTA per SM, although two run.)
__global__ void __launch_bounds__(kTcThreads) k_cluster_places(int* p) { if (p) *p = 0; }
static long long cluster_places(int n) {                          // n = 1, 2, 4 or 8
    constexpr int kSmem = 100 * 1024, kDevices = 64;
    static std::atomic<int> known[kDevices][4];                   // (asked on every launch: no lock)
    const int level = n == 8 ? 3 : n / 2;
    int dev = 0;
    if (n == 1 || cudaGetDevice(&dev) != cudaSuccess) return 2LL * sm_count() / n;
    const bool keep = dev >= 0 && dev < kDevices;
    int found = keep ? known[dev][level].load(std::memory_order_relaxed) : 0;
    if (found > 0) return found;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n); cfg.blockDim = dim3(kTcThreads); cfg.dynamicSmemBytes = kSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = n; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(k_cluster_places), kSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&found, k_cluster_places, &cfg) != cudaSuccess || found < 1) {
        cudaGetLastError();
        found = 2 * sm_count() / n;
    }
    if (keep) known[dev][level].store(found, std::memory_order_relaxed);
    return found;
}

// Chunks of a tile of `wy` rows in a launch over one clip: what split_of gives, but never fewer than tiles of one row have.
static int chunks_alone(const Problem& p, int wy, int sms) {
    const int own = own_chunks(tile_columns(p.r, wy)), one_row = split_of(p, (long long)tiles_of(p, 1), max_chunks(p.r), sms);
    int n = split_of(p, (long long)tiles_of(p, wy), max_chunks(p.r), sms);
    // (eight parts of 48 columns are not worth a second CTA on an SM: 5 x 29 x 13 x 1016 17.0 us per pass, with four 16.1)
    if (n > own && (long long)tiles_of(p, wy) * n > sms) n = own;
    return n > one_row ? n : one_row;
}
static int least_pieces(const Problem& p, int wy, int chunks) {           // (a CTA has tensor memory for own_chunks)
    const int own = own_chunks(tile_columns(p.r, wy));
    return chunks > own ? chunks / own : 1;
}
// Grid rows of a tile in a launch over `clips` clips, beside which nothing runs, whose channels are summed in `chunks` parts (0: as
// each tile has alone, and without a look at the places of clusters, which are not the same on every device).  The tile with the fewest rows to fetch, but not where its CTAs are more than one per SM and another tile's are done
// sooner: waves of two CTAs per SM x stages x rows of a stage.  Us per pass, replayed graph, the fewest rows / as here (CTAs):
// 40 x 26 x 20 x 1992 63.2 / 54.5 (175 / 195), 23 x 24 x 23 x 3856 63.5 / 58.0 (216 / 288), 40 x 32 x 32 x 2048 116.5 / 97.6 (320 / 384),
// 33 x 32 x 32 x 3000 144.3 / 119.7, 65 x 23 x 31 x 2216 131.3 / 114.6 (432 / 480), 20 x 20 x 20 x 2048 30.7 / 29.0 (with a fixed anchor
// 20.2 / 20.9), 54 x 30 x 19 x 2432 at r = 0 109.6 / 102.8 (300 / 280); three of 24 x 20 x 15 x 248 18.2 / 16.6.
static int tile_rows(const Problem& p, long long clips, int chunks, int sms) {
    const int nst = (p.C + kTcKC - 1) / kTcKC, few = fewest_rows(p);
    auto time = [&](int wy, long long* ctas) {
        const int n = chunks ? chunks : chunks_alone(p, wy, sms);
        const long long tiles = (long long)tiles_of(p, wy) * clips;
        int pieces = split_of(p, tiles, n, sms);
        while (chunks && pieces > 1 && tiles > cluster_places(pieces)) pieces /= 2;
        if (pieces < least_pieces(p, wy, n)) pieces = least_pieces(p, wy, n);
        *ctas = tiles * pieces;
        return (*ctas + 2 * sms - 1) / (2 * sms) * ((nst + pieces - 1) / pieces) * rows_per_stage(p, wy);
    };
    long long ctas, t[3] = {}, least = time(few, &ctas);
    if (ctas <= sms) return few;
    for (int i = 0; 1 << i <= most_rows(p); ++i) {
        t[i] = time(1 << i, &ctas);
        least = t[i] < least ? t[i] : least;
    }
    int best = 0;                                // the fewest rows among those that take at most a twentieth longer than the shortest
    for (int i = 0, wy = 1; wy <= most_rows(p); ++i, wy *= 2)
        if (t[i] * 20 <= least * 21 && (!best || tiles_of(p, wy) * rows_per_stage(p, wy) < tiles_of(p, best) * rows_per_stage(p, best))) best = wy;
    return best;
}

// How a launch splits its work.  The chunks depend on the clip's shape alone, the tile and its CTAs (= cluster size) on what is in
// flight.
TcPlan tc_plan(const Problem& p) {
    TcPlan t;
    // Three or more single clips in flight (ttf_set_schedule, clips that cannot share a launch)
    // fill the GPU together: 16 clips of 32 x 16 x 16 x 4096 on eight lanes 497 -> 445 us, on three 512 -> 506 (on two 530 ->
    // 507, but three clips, of which two share a launch, 98 -> 102).
    const int beside = p.nclips == 1 && p.overlapped >= 3 ? p.overlapped : 1;
    const int sms = sm_count();
    t.chunks = chunks_alone(p, tile_rows(p, 1, 0, sms), sms);
    // (beside another lane's kernels the fewest rows: 8 clips of 20 x 20 x 20 x 1024 73.4 us, by the rule above 80.4, 4 of
    // 40 x 16 x 16 x 1024 49.7 / 51.6, 2 of 23 x 24 x 23 x 2048 63.0 / 69.1.  The products of a row and a candidate are the same
    // whatever tile they are in.)
    t.rows = p.overlapped > 1 ? fewest_rows(p) : tile_rows(p, p.nclips, t.chunks, sms);
    t.tiles = (long long)tiles_of(p, t.rows);
    // Not more than run at the same time: the cluster that has to wait for a place costs the whole main loop once more (us per
    // pass, 32 frames of 2048 channels: 71 tiles in fours 23.4, 72 in fours 30.9, in twos 27.2; 33 in eights 19.6, 34 in
    // eights 23.8, in fours 20.6; 12 x 24 x 24 x 2048 28.8 -> 26.0).
    const long long units = t.tiles * p.nclips * beside;
    t.pieces = split_of(p, units, t.chunks, sms);
    while (t.pieces > 1 && units > cluster_places(t.pieces)) t.pieces /= 2;
    if (t.pieces < least_pieces(p, t.rows, t.chunks)) t.pieces = least_pieces(p, t.rows, t.chunks);
    return t;
}

template <int R, int WY, int G>
static cudaError_t launch_tc_t(const Problem& p, const TcPlan& plan, const Scratch& s, int* out_anchor, float* shat, int* dst,
                               unsigned char* keep, cudaStream_t st) {
    using S = TcShape<R, WY>;
    ClipMaps<G> maps;
    for (int n = 0; n < p.nclips; ++n)
        if (!make_tensor_map(&maps.a[n], p.xs.X[n], 1, p.F, p.H, p.W, p.C, kTcKC, kTcWB, WY, S::FR, true) ||
            !make_tensor_map(&maps.b[n], p.xs.X[n], 1, p.F, p.H, p.W, p.C, kTcKC, S::BW, S::BH, 1, true))
            return cudaErrorInvalidValue;
    // (at least 80 KB: never three CTAs on one SM while others have one or none; r = 0 would fit three)
    const size_t need = (size_t)S::RING + S::XBYTES + S::NORMBYTES + 1024, smem = need < 80 * 1024 ? 80 * 1024 : need;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_match_tc<R, WY, G>), smem);
    if (e != cudaSuccess) return e;
    const long long tiles = plan.tiles;
    const int chunks = plan.chunks, pieces = plan.pieces;
    auto log2_of = [](int n) { int l = 0; while ((1 << l) < n) ++l; return l; };
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * pieces), p.nclips); cfg.blockDim = dim3(kTcThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    int n = 1;
    if (pieces > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)pieces; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr; cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, k_match_tc<R, WY, G>, maps, p.F, p.H, p.W, p.C, p.t, make_anchor_src(p, s, out_anchor),
                              log2_of(pieces), log2_of(chunks), shat, dst, keep, s.cnt, wait_poll_limit(), wait_tx_extra(), p.stream_once, p.sstride, p.fuse_cnt);
}

template <int R, int G>
static cudaError_t launch_tc_rows(const Problem& p, const Scratch& s, int* out_anchor, float* shat, int* dst,
                                  unsigned char* keep, cudaStream_t st) {
    const TcPlan plan = tc_plan(p);
    if constexpr (R < 2) if (plan.rows == 4) return launch_tc_t<R, 4, G>(p, plan, s, out_anchor, shat, dst, keep, st);
    return plan.rows == 2 ? launch_tc_t<R, 2, G>(p, plan, s, out_anchor, shat, dst, keep, st)
                          : launch_tc_t<R, 1, G>(p, plan, s, out_anchor, shat, dst, keep, st);
}
template <int G>
static cudaError_t launch_tc(const Problem& p, const Scratch& s, int* out_anchor, float* shat, int* dst,
                             unsigned char* keep, cudaStream_t st) {
    if (p.r == 0) return launch_tc_rows<0, G>(p, s, out_anchor, shat, dst, keep, st);
    if (p.r == 1) return launch_tc_rows<1, G>(p, s, out_anchor, shat, dst, keep, st);
    return launch_tc_rows<2, G>(p, s, out_anchor, shat, dst, keep, st);
}
cudaError_t launch_match_tc(const Problem& p, const Scratch& s, int* out_anchor, float* shat, int* dst,
                            unsigned char* keep, cudaStream_t st) {
    return p.nclips > 1 ? launch_tc<kMaxGroup>(p, s, out_anchor, shat, dst, keep, st)
                        : launch_tc<1>(p, s, out_anchor, shat, dst, keep, st);
}

}  // namespace ttf
