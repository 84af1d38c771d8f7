// Extensions the paper sketches in its Discussion: TTF-R restoration through dst(k,i) (D4) and the empirical
// distribution of the best-match similarities that an adaptive threshold would look at (D1).
#include "ttf_internal.cuh"
#include "ttf_async.cuh"
#include "ttf_cluster.cuh"

#include <algorithm>

namespace ttf {

constexpr int kXThreads = 256;

// Number of non-zero flags in keep[lo, hi): bytes up to the first 16-byte boundary, 16 flags per load from there,
// bytes again at the end.  Every thread of the CTA takes part; the caller adds the per-thread counts up.  (Plain loads, as for
// the rows below: the CTAs of an SM read the same lines.  Past L1, restoring 128 x 32 x 32 tokens of 128 bytes took 24.5 us, 19.5 now.)
__device__ __forceinline__ int count_flags(const unsigned char* keep, size_t lo, size_t hi, int tid) {
    if (lo >= hi) return 0;
    int c = 0;
    const uintptr_t base = reinterpret_cast<uintptr_t>(keep);
    size_t head = lo + ((16 - ((base + lo) & 15)) & 15);          // first index whose address is 16-byte aligned
    if (head > hi) head = hi;
    const size_t nvec = (hi - head) / 16, tail = head + nvec * 16;
    for (size_t f = lo + tid; f < head; f += kXThreads) c += keep[f] ? 1 : 0;
    const uint4* v = reinterpret_cast<const uint4*>(keep + head);
    for (size_t u = tid; u < nvec; u += kXThreads) {
        const uint4 q = v[u];
        // a flag is any non-zero byte: fold each byte's bits into its lowest one
        unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            unsigned b = w[e];
            b |= b >> 4; b |= b >> 2; b |= b >> 1;
            c += __popc(b & 0x01010101u);
        }
    }
    for (size_t f = tail + tid; f < hi; f += kXThreads) c += keep[f] ? 1 : 0;
    return c;
}

// Row of the compressed sequence that stands for token (k,i): its own row if it was retained (anchor rows are
// rows 0..N-1, preserved source tokens follow in ascending flat order, Eq. xprime_stack), else the anchor row
// dst(k,i) it was fused into (Eq. dst).  One CTA per frame; it counts the flags of the frames before its own
// (16 per load, at most F N bytes, from L2 after the first CTA has touched them).
__global__ void __launch_bounds__(kXThreads)
k_restore_index(const int* __restrict__ anchor, const unsigned char* __restrict__ keep, const int* __restrict__ dst,
                int F, int N, int* __restrict__ row_index)
{
    __shared__ int s_warp[kXThreads / 32];
    __shared__ int s_base;
    pdl_launch_dependents();                     // the copy kernel may start its set-up; it waits before it reads row_index
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int a = *anchor;
    if (k == a) {
        for (int i = tid; i < N; i += kXThreads) row_index[(size_t)k * N + i] = i;
        return;
    }
    // preserved source tokens in the frames before this one (the anchor frame does not count)
    const size_t before = (size_t)k * N;
    int c = count_flags(keep, 0, before, tid);
    if (a >= 0 && a < k) c -= count_flags(keep, (size_t)a * N, (size_t)(a + 1) * N, tid);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) s_warp[w] = c;
    __syncthreads();
    if (tid == 0) { int b = 0; for (int ww = 0; ww < kXThreads / 32; ++ww) b += s_warp[ww]; s_base = b; }
    __syncthreads();
    int run = N + s_base;
    for (int i0 = 0; i0 < N; i0 += kXThreads) {
        const int i = i0 + tid;
        const bool kp = i < N && keep[before + i];
        const unsigned m = __ballot_sync(0xffffffffu, kp);
        __syncthreads();
        if (lane == 0) s_warp[w] = __popc(m);
        __syncthreads();
        int off = 0, total = 0;
        for (int ww = 0; ww < kXThreads / 32; ++ww) { if (ww < w) off += s_warp[ww]; total += s_warp[ww]; }
        if (i < N) row_index[before + i] = kp ? run + off + __popc(m & ((1u << lane) - 1)) : dst[before + i];
        run += total;
    }
}

// Rows f = first, first + step, ... < end of the output by one warp; `row(f)` is the compressed row that stands for token
// f.  A lane keeps up to eight loads in flight before it stores them, so a row of 8 KB moves in two rounds.  Rows of
// retained tokens are read once (consecutive tokens sit in consecutive compressed rows); the N anchor rows are read again
// and again and stay in L2.
template <typename U, typename Row>
__device__ __forceinline__ void restore_rows(const unsigned char* comp, size_t row_bytes, long long first,
                                             long long end, long long step, unsigned char* out, int lane,
                                             Row&& row) {
    constexpr int kInFlight = 8;
    const int units = (int)(row_bytes / sizeof(U));
    for (long long f = first; f < end; f += step) {
        const U* src = reinterpret_cast<const U*>(comp + (size_t)row(f) * row_bytes);
        U* d = reinterpret_cast<U*>(out + (size_t)f * row_bytes);
        int u = lane;
        for (; u + (kInFlight - 1) * 32 < units; u += kInFlight * 32) {
            U v[kInFlight];
#pragma unroll
            for (int e = 0; e < kInFlight; ++e) v[e] = src[u + e * 32];
#pragma unroll
            for (int e = 0; e < kInFlight; ++e) d[u + e * 32] = v[e];
        }
        for (; u < units; u += 32) d[u] = src[u];
    }
}

template <typename U>
__global__ void __launch_bounds__(kXThreads)
k_restore_copy(const unsigned char* __restrict__ comp, size_t row_bytes, long long rows,
               const int* __restrict__ row_index, unsigned char* __restrict__ out)
{
    const long long gw = (long long)blockIdx.x * (kXThreads / 32) + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * (kXThreads / 32);
    pdl_wait();                                  // row_index is complete
    restore_rows<U>(comp, row_bytes, gw, rows, nw, out, threadIdx.x & 31, [&](long long f) { return __ldcg(row_index + f); });
}

// The compressed rows of tokens [f0, f1), which belong to this CTA: it counts the preserved tokens before them (16 flags per load:
// one round trip) and ranks its own, 256 at a time; round(b0, end) finds the rows of tokens [b0, end) in s_row.  The anchor
// frame's tokens are [a0, a1), none of the clip's for an anchor outside it.
template <typename Round>
__device__ __forceinline__ void restore_rounds(int FN, int N, const int* anchor, const unsigned char* keep, const int* dst, int f0, int f1,
                                               int* row_index, int* s_warp, int* s_row, Round&& round) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // (what the first round needs of this CTA's tokens is asked for together with the anchor and the flags before them)
    unsigned char next_keep = f0 + tid < f1 ? keep[f0 + tid] : (unsigned char)0;
    int next_dst = f0 + tid < f1 ? dst[f0 + tid] : 0;
    const int a = __ldcg(anchor);
    const bool inside = (unsigned)a < (unsigned)(FN / N);
    const int a0 = inside ? a * N : FN, a1 = inside ? a0 + N : FN;
    int c = count_flags(keep, 0, (size_t)min(f0, a0), tid);      // (the anchor frame does not count)
    if (f0 > a1) c += count_flags(keep, (size_t)a1, (size_t)f0, tid);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) s_warp[w] = c;
    __syncthreads();
    int run = N;
#pragma unroll
    for (int ww = 0; ww < kXThreads / 32; ++ww) run += s_warp[ww];
    for (int b0 = f0; b0 < f1; b0 += kXThreads) {
        const int f = b0 + tid;
        const bool in = f < f1, own = f >= a0 && f < a1;
        const bool kp = in && !own && next_keep;
        const int to = next_dst;
        next_keep = f + kXThreads < f1 ? keep[f + kXThreads] : (unsigned char)0;
        next_dst = f + kXThreads < f1 ? dst[f + kXThreads] : 0;
        const unsigned m = __ballot_sync(0xffffffffu, kp);
        __syncthreads();                         // (the indices of the round before this one, and s_warp, are done with)
        if (lane == 0) s_warp[w] = __popc(m);
        __syncthreads();
        int off = 0, total = 0;
#pragma unroll
        for (int ww = 0; ww < kXThreads / 32; ++ww) { off += ww < w ? s_warp[ww] : 0; total += s_warp[ww]; }
        if (in) {
            const int r = own ? f - a0 : (kp ? run + off + __popc(m & ((1u << lane) - 1)) : to);
            s_row[tid] = r;
            row_index[f] = r;
        }
        run += total;
        __syncthreads();
        round(b0, min(f1, b0 + kXThreads));
    }
}

// Both steps in one launch, for clips of up to kRestoreWhole tokens: a CTA owns a contiguous range of tokens and copies their rows
// from the indices in shared memory.  What bounds it is the traffic of long rows, and for short ones a chain of round trips.  Us
// per call / in a replayed graph, with a launch for the indices -> in one: 4 x 16 x 16 x 64 bf16 channels 11.7 / 3.9 -> 8.9 /
// 2.4, 32 x 16 x 16 x 64 11.7 / 4.9 -> 8.7 / 6.3, 32 x 16 x 16 x 4096 18.5 / 16.9 -> 15.3 / 15.2 (its 90 MB at the copy rate:
// 13.8), 64 x 32 x 32 x 64 15.4 / 13.0 -> 14.1 / 14.0, x 1024 53.7 / 48.7 -> 45.5 / 45.4: the graph's time alone would draw the
// line for short rows at 4096 tokens, a call's at 65536.  In longer clips the flags that every CTA reads outweigh the launch.
constexpr int kRestoreWhole = 1 << 16;

template <typename U>
__global__ void __launch_bounds__(kXThreads)
k_restore(const unsigned char* comp, size_t row_bytes, int FN, int N, const int* anchor, const unsigned char* keep,
          const int* dst, int per, unsigned char* out, int* row_index)
{
    __shared__ int s_warp[kXThreads / 32];
    __shared__ int s_row[kXThreads];
    const int f0 = blockIdx.x * per, f1 = min(FN, f0 + per);
    pdl_launch_dependents();
    pdl_wait();                                  // the caller's kernels before this one
    restore_rounds(FN, N, anchor, keep, dst, f0, f1, row_index, s_warp, s_row, [&](int b0, int end) {
        restore_rows<U>(comp, row_bytes, b0 + (threadIdx.x >> 5), end, kXThreads / 32, out, threadIdx.x & 31,
                        [&](long long g) { return s_row[(int)g - b0]; });
    });
}

// The same with bulk copies, for rows of whole 16-byte pieces: one CTA per SM (see restore_plan), whose warps move batches of
// consecutive output rows (or pieces of long ones) through three slots, two loads ahead; a batch leaves as one store.  The flags
// before a CTA's tokens are read by 148 CTAs instead of up to 1184 (they queue on the same lines), short rows move 32 to a batch, and a
// row that is no multiple of eight loads per lane has no serial rest.  Us per call in a replayed graph, plain loads / bulk:
// 32 x 16 x 16 x 512 7.2 / 4.9, 64 x 32 x 32 x 64 14.4 / 8.3, 14 x 25 x 14 x 2800 13.9 / 9.8, 48 x 16 x 16 x 1536 21.6 / 12.0,
// 64 x 32 x 32 x 1024 47.8 / 36.3; from two launches 128 x 32 x 32 x 64 27.8 / 15.9, x 512 53.3 / 38.7, 256 x 32 x 32 x 64 50.1 /
// 30.0.  (Two slots of 8 KB 10.2 and 12.4 where three take 9.8 and 12.0; four of 4 KB 10.9.)
// A wait that runs out has nobody to report to here: the warp copies what is left by plain loads and stores.
constexpr int kRestoreBulk = 1 << 18;
constexpr int kRestoreSlots = 3, kRestoreAhead = 2;
__global__ void __launch_bounds__(kXThreads)
k_restore_bulk(const unsigned char* comp, size_t row_bytes, int FN, int N, const int* anchor, const unsigned char* keep,
               const int* dst, int per, unsigned char* out, int* row_index, int pieces, int batch, int slots, int slot, int wait_limit, int tx_extra)
{
    extern __shared__ __align__(128) unsigned char stage[];      // [warps][slots][slot]
    __shared__ uint64_t bar[kXThreads / 32][kRestoreSlots];
    __shared__ int s_warp[kXThreads / 32];
    __shared__ int s_row[kXThreads];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int f0 = blockIdx.x * per, f1 = min(FN, f0 + per);
    pdl_launch_dependents();
    if (lane == 0) {
        for (int h = 0; h < kRestoreSlots; ++h) mbar_init(&bar[w][h], 1);
        mbar_init_fence();
    }
    __syncwarp();
    pdl_wait();                                  // the caller's kernels before this one
    unsigned char* const buf = stage + (size_t)w * slots * slot;
    int issued = 0, finished = 0;                // batches of this warp; batch n goes through slot n % kRestoreSlots
    bool gave_up = false;
    restore_rounds(FN, N, anchor, keep, dst, f0, f1, row_index, s_warp, s_row, [&](int b0, int end) {
        const int R = max(1, min(batch, (end - b0 + kXThreads / 32 - 1) / (kXThreads / 32)));
        const int units = (end - b0) * pieces, step = kXThreads / 32 * R;
        auto piece_bytes = [&](int pc) { return (uint32_t)min(row_bytes - (size_t)pc * slot, (size_t)slot); };
        auto issue = [&](int u) {
            const int n = min(R, units - u), h = issued % kRestoreSlots;
            const int r0 = pieces == 1 ? u : u / pieces, pc = pieces == 1 ? 0 : u - r0 * pieces;
            if (lane == 0) {
                bulk_wait_read<kRestoreSlots - 1 - kRestoreAhead>();      // the store that used this slot has finished reading it
                mbar_arrive_expect_tx(&bar[w][h], (uint32_t)n * piece_bytes(pc) + (uint32_t)tx_extra);
            }
            __syncwarp();
            if (lane < n)
                bulk_load(buf + h * slot + lane * (uint32_t)row_bytes,
                          comp + (size_t)s_row[r0 + lane] * row_bytes + (size_t)pc * slot, piece_bytes(pc), &bar[w][h]);
            ++issued;
        };
        int ahead = w * R;
        for (int q = 0; q < kRestoreAhead && ahead < units && !gave_up; ++q, ahead += step) issue(ahead);
        for (int u = w * R; u < units; u += step) {
            const int n = min(R, units - u);
            const int r0 = pieces == 1 ? u : u / pieces, pc = pieces == 1 ? 0 : u - r0 * pieces;
            unsigned char* d = out + (size_t)(b0 + r0) * row_bytes + (size_t)pc * slot;
            if (!gave_up) {
                if (ahead < units) { issue(ahead); ahead += step; }
                const int h = finished % kRestoreSlots;
                bool ok = true;
                if (lane == 0) ok = mbar_wait(&bar[w][h], (finished / kRestoreSlots) & 1, wait_limit);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (ok) {
                    if (lane == 0) {
                        bulk_store(d, buf + h * slot, (uint32_t)n * piece_bytes(pc));
                        bulk_commit();
                    }
                    ++finished;
                    continue;
                }
                gave_up = true;
            }
            // a copy that does not arrive: this batch and the rest by plain loads and stores
            for (int q = 0; q < n; ++q) {
                const uint4* src = reinterpret_cast<const uint4*>(comp + (size_t)s_row[r0 + q] * row_bytes + (size_t)pc * slot);
                uint4* to4 = reinterpret_cast<uint4*>(d + (size_t)q * row_bytes);
                for (int e = lane; e < (int)(piece_bytes(pc) / 16); e += 32) to4[e] = src[e];
            }
        }
    });
    if (lane == 0) {
        // copies still on their way into this CTA's shared memory (bounded again)
        for (; finished < issued; ++finished) mbar_wait(&bar[w][finished % kRestoreSlots], (finished / kRestoreSlots) & 1, wait_limit);
        bulk_wait<0>();
    }
}

template <typename U>
static cudaError_t launch_restore_t(const unsigned char* c, size_t row_bytes, int F, int N, const int* anchor,
                                    const unsigned char* keep, const int* dst, unsigned char* o, int* row_index,
                                    cudaStream_t st) {
    const long long rows = (long long)F * N;
    long long blocks = (rows + kXThreads / 32 - 1) / (kXThreads / 32);
    if (blocks > 8LL * sm_count()) blocks = 8LL * sm_count();
    if (rows <= kRestoreWhole) {
        const int per = (int)((rows + blocks - 1) / blocks);
        return launch_pdl(k_restore<U>, dim3((unsigned)((rows + per - 1) / per)), dim3(kXThreads), st, c, row_bytes, (int)rows,
                          N, anchor, keep, dst, per, o, row_index);
    }
    k_restore_index<<<F, kXThreads, 0, st>>>(anchor, keep, dst, F, N, row_index);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_pdl(k_restore_copy<U>, dim3((unsigned)blocks), dim3(kXThreads), st, c, row_bytes, rows, row_index, o);
}

// How a call copies, by size.  Calls on other streams of the caller's want room on the SMs too, and with 192 KB of slots in every
// launch two restores cannot share an SM.  Us per call in a replayed graph, on one / two / four streams:
//                           plain loads             192 KB of slots         as here
//   5 x 16 x 16 x  512       2.96   1.67   1.19      3.05   2.40   2.37      (plain)
//   9 x 16 x 16 x 1024       5.91   3.41   2.63      4.04   3.04   3.04      4.39   2.70   1.85
//  12 x 16 x 16 x 2048       5.81   3.80   3.16      5.72   4.41   4.43      (plain)
//  20 x 16 x 16 x 2048       8.36   5.58   4.92      7.24   5.84   5.78      7.36   5.49   5.46
//  32 x 16 x 16 x 2048      10.74   7.48   7.52      9.93   8.24   7.99     10.13   7.74   7.50
//  16 x 16 x 16 x 1024       6.76   4.22   4.00      4.88   3.87   3.86      (192 KB)
//  64 x 16 x 16 x 1024      17.5   12.5   12.5      10.2    8.6    8.4       (192 KB)
//  - Rows of whole 4 KB keep eight plain loads per lane in flight throughout and gain from bulk copies only between 20 and 52 MB of
//    output (bulk / plain alone: 50 MB 15.1 / 15.3, 67 MB in rows of 4 KB 19.0 / 18.3, of 8 KB 19.0 / 18.0, 151 MB 41.9 / 37.6);
//    there two CTAs of 96 KB per SM do as well as one of 192 KB.
//  - The smallest clips gain nothing from the way through shared memory (131 KB 3.65 / 3.15, 524 KB 3.65 / 3.4, in 4096 rows 3.66 /
//    4.15).
//  - Clips of up to 3072 tokens take no more slots, and no larger ones, than their warps fill; from about there on plain loads were
//    never the faster ones.
struct RestorePlan { bool bulk; int ctas, per, pieces, batch, slots, slot; size_t smem; };
static RestorePlan restore_plan(long long FN, size_t row_bytes) {
    constexpr int warps = kXThreads / 32;
    const double mb = (double)FN * row_bytes * 1e-6;
    const bool whole_4k = row_bytes % 4096 == 0;
    RestorePlan q = {};
    q.bulk = FN <= kRestoreBulk && (whole_4k ? mb > 20.0 && mb <= 52.0 : FN > 2048 || mb > 1.5);
    if (!q.bulk) return q;
    const size_t most = whole_4k ? 4096 : 8192;              // bytes of a slot
    const int ctas = sm_count() * (whole_4k ? 2 : 1);
    q.per = (int)std::max<long long>(warps, (FN + ctas - 1) / ctas);
    q.ctas = (int)((FN + q.per - 1) / q.per);
    q.pieces = (int)((row_bytes + most - 1) / most);
    q.batch = q.pieces > 1 ? 1 : (int)std::min<size_t>(32, most / row_bytes);
    q.slots = kRestoreSlots;
    q.slot = (int)most;
    if (FN <= 3072 && q.per <= kXThreads) {      // (one round)
        const int rows = (q.per + warps - 1) / warps;
        if (q.pieces == 1) {
            q.batch = std::min(q.batch, rows);
            q.slot = (int)(q.batch * row_bytes);
        }
        q.slots = (int)std::min<long long>(kRestoreSlots, ((long long)rows * q.pieces + q.batch - 1) / q.batch);
    }
    q.smem = (size_t)warps * q.slots * q.slot;
    return q;
}

cudaError_t launch_restore(const void* comp, size_t row_bytes, int F, int N, const int* anchor,
                           const unsigned char* keep, const int* dst, void* out_full, int* row_index,
                           cudaStream_t st) {
    const unsigned char* c = reinterpret_cast<const unsigned char*>(comp);
    unsigned char* o = reinterpret_cast<unsigned char*>(out_full);
    const uintptr_t al = reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(out_full) | row_bytes;
    const RestorePlan q = restore_plan((long long)F * N, row_bytes);
    if (al % 16 == 0 && q.bulk) {
        cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_restore_bulk), q.smem);
        if (e != cudaSuccess) return e;
        return launch_ex(true, q.smem, k_restore_bulk, dim3(q.ctas), dim3(kXThreads), st, c, row_bytes, F * N, N, anchor, keep,
                         dst, q.per, o, row_index, q.pieces, q.batch, q.slots, q.slot, wait_poll_limit(), wait_tx_extra());
    }
    if (al % 16 == 0) return launch_restore_t<uint4>(c, row_bytes, F, N, anchor, keep, dst, o, row_index, st);
    if (al % 4 == 0) return launch_restore_t<uint32_t>(c, row_bytes, F, N, anchor, keep, dst, o, row_index, st);
    if (al % 2 == 0) return launch_restore_t<uint16_t>(c, row_bytes, F, N, anchor, keep, dst, o, row_index, st);
    return launch_restore_t<unsigned char>(c, row_bytes, F, N, anchor, keep, dst, o, row_index, st);
}

// Histogram of the best-match similarities of the source tokens over `bins` equal bins of [-1, 1]
// (bin = floor((s + 1) / 2 * bins), clamped; NaN is not counted).  Integer atomics: order-independent.
__global__ void __launch_bounds__(kXThreads)
k_sim_histogram(const float* __restrict__ sim, const int* __restrict__ anchor, int N, long long total, int bins,
                unsigned int* __restrict__ hist)
{
    const int a = *anchor;
    const long long stride = (long long)gridDim.x * kXThreads;
    for (long long f = (long long)blockIdx.x * kXThreads + threadIdx.x; f < total; f += stride) {
        if (f / N == a) continue;
        const float s = sim[f];
        if (!(s == s)) continue;
        int b = (int)floorf((s + 1.0f) * 0.5f * (float)bins);
        b = b < 0 ? 0 : (b >= bins ? bins - 1 : b);
        atomicAdd(&hist[b], 1u);
    }
}

cudaError_t launch_sim_histogram(const float* sim, const int* anchor, int F, int N, int bins, unsigned int* hist,
                                 cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned int) * (size_t)bins, st);
    if (e != cudaSuccess) return e;
    const long long total = (long long)F * N;
    long long blocks = (total + kXThreads - 1) / kXThreads;
    if (blocks > 4LL * sm_count()) blocks = 4LL * sm_count();
    k_sim_histogram<<<(unsigned)blocks, kXThreads, 0, st>>>(sim, anchor, N, total, bins, hist);
    return cudaGetLastError();
}

// Counts behind the reduction ratio rho = 1 - (N + P) / (F N) (Sec. 3, after Eq. Lpre) and the number of source
// tokens whose best similarity lies within `band` of the threshold (the decisions rounding could flip).
// out[0] = P (preserved source tokens), out[1] = fused source tokens, out[2] = in-band source tokens.  The band test
// is taken in double on the stored fp32 values, so the counts are exact functions of the arrays.  Integer atomics.
struct TokenCounts { int c[3]; };                // P, fused, in band

__device__ __forceinline__ void count_token(TokenCounts& n, bool source, bool kept, float sim, float t, float band) {
    n.c[0] += source && kept;
    n.c[1] += source && !kept;
    n.c[2] += source && fabs((double)sim - (double)t) < (double)band;
}
// sums over the CTA, to threads 0 .. 2 (count i in thread i); s_part: [3][warps]
template <int WARPS> __device__ __forceinline__ int counts_of_block(TokenCounts& n, int (&s_part)[3][WARPS]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n.c[q] += __shfl_xor_sync(0xffffffffu, n.c[q], o);
        if (lane == 0) s_part[q][w] = n.c[q];
    }
    __syncthreads();
    int v = 0;
    if (threadIdx.x < 3)
        for (int ww = 0; ww < WARPS; ++ww) v += s_part[threadIdx.x][ww];
    return v;
}

// Clips of up to kStatsWhole tokens: one cluster of eight CTAs, whose counts meet in the shared memory of rank 0.  (A grid
// of independent CTAs needs its three words cleared first: a memset before the kernel, 5 us of 37 for the query and the
// counts of a 48 x 14 x 14 clip of 2048 channels.)  The cluster's time grows with the clip, us in a replayed graph, cluster /
// grid: 9408 tokens 1.9 / 5.9, 98304 3.5 / 5.9, 196608 5.5 / 5.9, 262144 6.6 / 6.2.
constexpr int kStatsCtas = 8, kStatsThreads = 512;
constexpr long long kStatsWhole = 3 << 16;

__global__ void __cluster_dims__(kStatsCtas, 1, 1) __launch_bounds__(kStatsThreads)
k_stats_cluster(const float* sim, const unsigned char* keep, const int* anchor, int N, int total, float t, float band,
                long long* out)
{
    __shared__ int s_part[3][kStatsThreads / 32];
    __shared__ int s_in[kStatsCtas][3];
    pdl_launch_dependents();
    cluster_arrive();                            // this CTA runs: the others may write into it
    pdl_wait();                                  // (what the kernel before this one wrote is read with L2-coherent loads)
    const int a = __ldcg(anchor);                // (outside the clip: no token is the anchor frame's)
    const bool inside = (unsigned)a < (unsigned)(total / N);
    const int a0 = inside ? a * N : 0, a1 = inside ? a0 + N : 0;
    const int rank = (int)cluster_rank();
    TokenCounts n = {{0, 0, 0}};
    constexpr int kInFlight = 4, kStride = kStatsCtas * kStatsThreads;
    for (int f0 = rank * kStatsThreads + (int)threadIdx.x; f0 < total; f0 += kInFlight * kStride) {
        unsigned char kp[kInFlight];
        float s[kInFlight];
#pragma unroll
        for (int u = 0; u < kInFlight; ++u) {
            const int f = min(f0 + u * kStride, total - 1);
            kp[u] = __ldcg(keep + f);
            s[u] = __ldcg(sim + f);
        }
#pragma unroll
        for (int u = 0; u < kInFlight; ++u) {
            const int f = f0 + u * kStride;
            count_token(n, f < total && (f < a0 || f >= a1), kp[u] != 0, s[u], t, band);
        }
    }
    const int v = counts_of_block(n, s_part);
    __syncwarp();
    cluster_wait();                              // every CTA has started
    if (threadIdx.x < 3) st_cluster_u32(cluster_addr(smem_u32(&s_in[rank][threadIdx.x]), 0), (uint32_t)v);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (rank == 0 && threadIdx.x < 3) {
        long long sum = 0;
#pragma unroll
        for (int r = 0; r < kStatsCtas; ++r) sum += s_in[r][threadIdx.x];
        out[threadIdx.x] = sum;
    }
}

__global__ void __launch_bounds__(kXThreads)
k_stats(const float* __restrict__ sim, const unsigned char* __restrict__ keep, const int* __restrict__ anchor, int N,
        long long total, float t, float band, unsigned long long* __restrict__ out)
{
    __shared__ int s_part[3][kXThreads / 32];
    const int a = *anchor;
    TokenCounts n = {{0, 0, 0}};
    const long long stride = (long long)gridDim.x * kXThreads;
    for (long long f = (long long)blockIdx.x * kXThreads + threadIdx.x; f < total; f += stride)
        count_token(n, f / N != a, keep[f] != 0, sim[f], t, band);
    const int v = counts_of_block(n, s_part);
    if (threadIdx.x < 3 && v) atomicAdd(out + threadIdx.x, (unsigned long long)v);
}

cudaError_t launch_stats(const float* sim, const unsigned char* keep, const int* anchor, int F, int N, float t, float band,
                         long long* out, cudaStream_t st) {
    const long long total = (long long)F * N;
    if (total <= kStatsWhole)
        return launch_pdl(k_stats_cluster, dim3(kStatsCtas), dim3(kStatsThreads), st, sim, keep, anchor, N, (int)total, t, band,
                          out);
    cudaError_t e = cudaMemsetAsync(out, 0, 3 * sizeof(long long), st);
    if (e != cudaSuccess) return e;
    long long blocks = (total + kXThreads - 1) / kXThreads;
    if (blocks > 2LL * sm_count()) blocks = 2LL * sm_count();
    k_stats<<<(unsigned)blocks, kXThreads, 0, st>>>(sim, keep, anchor, N, total, t, band,
                                                   reinterpret_cast<unsigned long long*>(out));
    return cudaGetLastError();
}

// Measurement aid: the plainest kernel that reads a buffer once (fully coalesced, eight 16-byte loads in flight per
// thread, eight CTAs of 256 threads per SM, launched like the kernels of the pass).  What a launch of this kind
// takes on one clip is the floor for any kernel that must read that clip: ramp-up and tail of a launch that lasts
// some 10 us are a visible share of it, so it is well below the copy rate of large buffers.
__global__ void __launch_bounds__(kXThreads)
k_read_floor(const uint4* __restrict__ buf, long long n16, unsigned* __restrict__ sink)
{
    pdl_launch_dependents();
    pdl_wait();
    unsigned acc = 0;
    const long long stride = (long long)gridDim.x * kXThreads * 8;
    for (long long i0 = (long long)blockIdx.x * kXThreads * 8 + threadIdx.x; i0 < n16; i0 += stride) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i0 + u * kXThreads < n16 ? __ldcs(buf + i0 + u * kXThreads) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += v[u].x ^ v[u].y ^ v[u].z ^ v[u].w;
    }
    if (acc == 0x9e3779b9u && sink) *sink = acc;       // keeps the loads alive; practically never true
}

cudaError_t launch_read_floor(const void* buf, size_t bytes, unsigned* sink, cudaStream_t st) {
    return launch_pdl(k_read_floor, dim3((unsigned)(8 * sm_count())), dim3(kXThreads), st,
                      reinterpret_cast<const uint4*>(buf), (long long)(bytes / 16), sink);
}

}  // namespace ttf
