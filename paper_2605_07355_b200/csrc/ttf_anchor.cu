// Anchor Frame Selection (Eq. auto_anchor) and per-token norms: one streaming sweep over X plus a small
// statistics kernel whose last CTA takes the arg max (resolve_anchor).
//
// k_norm_sum.  A CTA owns (frame k, channel slice q); a slice is LS lanes x one 16-byte load (512 bytes
// of every token row with LS = 32, less where a clip would make too few CTAs; the CTAs of neighbouring slices run side by
// side, so DRAM sees whole rows).  The
// 256 / LS row groups of a CTA walk the tokens of the frame interleaved, eight tokens per thread in
// flight and the next eight prefetched.  A thread keeps running sums of its channels; the row groups are combined through
// shared memory in a fixed order and give the frame sum S_k[slice] (= N x mean token of frame k) directly.
// The squared norm of every token restricted to one warp's 32 lanes is reduced with a 9-shuffle fold and
// stored as a partial (consumers add the partials in plane order).
//
// k_frame_stats.  One CTA per 128-channel slice forms g[slice] = sum_k S_k[slice] and the slice's shares of
// <S_k, g>, |S_k|^2 and |g|^2 (the factors 1/N and 1/(FN) of Eq. auto_anchor cancel in a cosine).  Every order
// of summation is fixed, so the result is reproducible.
#include "ttf_internal.cuh"
#include "ttf_async.cuh"
#include "ttf_cluster.cuh"

#include <map>
#include <mutex>
#include <set>
#include <utility>

namespace ttf {

constexpr int kNormWarps = 8;
constexpr int kNormThreads = kNormWarps * 32;
constexpr int kBatch = 8;            // tokens per thread in flight (times two with the prefetch)

// Sum of v[u] over the warp for u = 0..7 with 9 shuffles.  On return the lanes with (lane & 3) == 0 hold the
// total of token u = 4*bit4 + 2*bit3 + bit2 of their lane index.
__device__ __forceinline__ float fold8(float (&v)[8], int lane) {
    {
        const bool up = lane & 16;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float send = up ? v[j] : v[j + 4];
            const float keep = up ? v[j + 4] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
    }
    {
        const bool up = lane & 8;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float send = up ? v[j] : v[j + 2];
            const float keep = up ? v[j + 2] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
    }
    {
        const bool up = lane & 4;
        const float send = up ? v[0] : v[1];
        const float keep = up ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    float r = v[0];
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}

// LS: lanes across a slice (8, 16 or 32); RG = 256 / LS row groups walk the tokens interleaved.
// CLS: a thread keeps CLS running sums, of every CLS-th of its tokens.  A sum over all tokens is the same tree whether 32
// classes of tokens belong to 32 row groups of 8 lanes (CLS = 1), to 16 of 16 (2) or to 8 of 32 (4): class w + 8 J to warp w,
// the J = 0..3 of a warp as (0 + 1) + (2 + 3), then the warps in order; likewise 16 classes.
// NORMS: also store the per-token partial squared norms (only the CUDA-core matching kernel reads them).
template <typename T, int V, int LS, bool NORMS, int CLS>
__global__ void __launch_bounds__(kNormThreads)
k_norm_sum(const __grid_constant__ ClipPtrs xs, int F, int N, int C, int nq,
           float* __restrict__ S, float* __restrict__ ssq, int* __restrict__ cnt, int* __restrict__ hdr,
           int flags, size_t sstride)
{
    const bool chain = flags & 1;                   // (bit 0: chain, bit 1: fresh; see Problem)
    const T* __restrict__ X = reinterpret_cast<const T*>(xs.X[blockIdx.y]);
    S = clip_block(S, sstride); ssq = clip_block(ssq, sstride); cnt = clip_block(cnt, sstride); hdr = clip_block(hdr, sstride);
    using L = Loader<T, V>;
    constexpr int RG = kNormThreads / LS;
    pdl_launch_dependents();
    // This kernel may be scheduled while the kernel before it in the stream still runs.  Normally that kernel may be
    // anything (the previous call's gather, which shares the scratch, or an upstream kernel that still writes X), so
    // nothing is read or written before the wait.  Inside a chain of clips of one batch the predecessor is known: the
    // gather of the previous clip, which works on another scratch block and another clip; then the sweep runs beside
    // it, and one CTA waits for it before it exits, so that "this sweep has completed" still implies "everything
    // before it has completed" for the kernels that follow.  (One CTA, not all: a CTA that waits keeps its place on
    // the SM, and the CTAs of the sweep that have not started yet need those places.)
    if (!chain) pdl_wait();
    trace_mark(hdr, 0, false);
    if (chain) trace_mark(hdr, 15, false);
    const int k = blockIdx.x / nq, q = blockIdx.x - k * nq;
    const int tid = threadIdx.x, lane = tid & 31;
    const int ls = tid & (LS - 1), rg = (tid >> 5) + kNormWarps * (lane / LS);
    const size_t FN = (size_t)F * N;
    const int c0 = (q * LS + ls) * V;
    const bool active = c0 < C;                     // C is a multiple of V on the vector path
    const T* base = X + (size_t)k * N * C + c0;
    float* plane = ssq + (size_t)q * FN + (size_t)k * N;           // (NORMS: LS = 32, one plane per slice)

    __shared__ float sm[kNormWarps][LS * V];
    static_assert(kBatch % CLS == 0, "whole rounds of the classes");
    float col[CLS][V];
#pragma unroll
    for (int c = 0; c < CLS; ++c)
#pragma unroll
        for (int v = 0; v < V; ++v) col[c][v] = 0.f;

    // thread's tokens: rg, rg + RG, rg + 2 RG, ...; a batch is kBatch of them
    typename L::Raw cur[kBatch], nxt[kBatch];
    auto load_batch = [&](typename L::Raw (&d)[kBatch], int i0) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = i0 + u * RG;
            d[u] = (active && i < N) ? L::load_raw_cg(base + (size_t)i * C) : L::zero();
        }
    };
    if (rg < N) load_batch(cur, rg);
    for (int i0 = rg; i0 < N; i0 += RG * kBatch) {
        if (i0 + RG * kBatch < N) load_batch(nxt, i0 + RG * kBatch);
        float ss[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            float x[V];
            L::unpack(cur[u], x);
            float s = 0.f;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (NORMS) s = fmaf(x[v], x[v], s);
                col[u % CLS][v] += x[v];
            }
            ss[u] = s;
        }
        if (NORMS) {
#pragma unroll
            for (int h = 0; h < kBatch / 8; ++h) {
                float part[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) part[e] = ss[h * 8 + e];
                const float tot = fold8(part, lane);
                const int u = h * 8 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
                if ((lane & 3) == 0 && i0 + u * RG < N) plane[i0 + u * RG] = tot;
            }
        }
#pragma unroll
        for (int uu = 0; uu < kBatch; ++uu) cur[uu] = nxt[uu];
    }

#pragma unroll
    for (int o = LS; o < 32; o <<= 1)               // the row groups of a warp (the low bits of J)
#pragma unroll
        for (int c = 0; c < CLS; ++c)
#pragma unroll
            for (int v = 0; v < V; ++v) col[c][v] += __shfl_xor_sync(0xffffffffu, col[c][v], o);
#pragma unroll
    for (int v = 0; v < V; ++v) {                   // and of a thread (the high bits)
        if (CLS == 2) col[0][v] += col[CLS / 2][v];
        if (CLS == 4) col[0][v] = (col[0][v] + col[CLS / 4][v]) + (col[CLS / 2][v] + col[CLS - 1][v]);
    }
    if (lane < LS) {
#pragma unroll
        for (int v = 0; v < V; ++v) sm[tid >> 5][ls * V + v] = col[0][v];
    }
    __syncthreads();
    for (int idx = tid; idx < LS * V; idx += kNormThreads) {
        const int c = q * LS * V + idx;
        if (c < C) {
            float s = 0.f;
#pragma unroll
            for (int r2 = 0; r2 < kNormWarps; ++r2) s += sm[r2][idx];
            if (in_bounds(hdr, 1, (long long)k * C + c, (long long)F * C)) S[(size_t)k * C + c] = s;
        }
    }
    if (q == 0 && tid == 0) cnt[k] = 0;             // survivor counters start at zero for the matching kernel
    if (blockIdx.x == 0 && tid == 0) clear_words(hdr, flags & 2);
    if (chain && blockIdx.x == 0 && blockIdx.y == 0) pdl_wait();
    trace_mark(hdr, 0, true);
}

template <typename T, int V, int LS, bool NORMS, int CLS = 1>
static cudaError_t launch_sum_ls(const Problem& p, const Scratch& s, cudaStream_t st) {
    const int nq = (p.C + LS * V - 1) / (LS * V);
    return launch_ex(true, 0, k_norm_sum<T, V, LS, NORMS, CLS>, dim3((unsigned)((long long)p.F * nq), p.nclips), dim3(kNormThreads),
                     st, p.xs, p.F, p.N, p.C, nq, s.S, s.ssq, s.cnt, s.hdr, p.chain | (p.fresh << 1), p.sstride);
}

template <typename T, int V>
static cudaError_t launch_sum_t(const Problem& p, const Scratch& s, cudaStream_t st) {
    if (needs_sweep_norms(p)) return launch_sum_ls<T, V, 32, true>(p, s, st);
    // Width of a slice: a warp across (512 bytes of a row), unless the launch then has fewer than two CTAs per SM: half or a
    // quarter of a warp, with as many more rows in flight per warp.  Us per pass, 32 lanes / at most 16 / at most 8 / at most
    // 4: 4 x 32 x 32 x 256 21.7 / 17.8 / 15.9 / 14.7, 4 x 32 x 32 x 1024 28.0 / 25.2 / 22.6 / 22.3, 8 x 24 x 24 x 2048
    // 31.7 / 28.1 / 26.4 / 28.6, 32 x 16 x 16 x 1024 20.7 / 19.2 / 18.2 / 18.3, 16 x 8 x 8 x 512 12.2 / 12.5 / 12.3 / 12.8;
    // with 512 CTAs as they are (32 x 16 x 16 x 4096) narrower slices gain nothing (37.9 / 38.2), and a batch of eight
    // 24 x 20 x 20 x 1024 has enough of them together (86.4 against 89.9 with narrow slices).
    // The order of summation is that of the width which the clip takes alone, so that the anchor does not depend on the launch:
    // wider slices keep the sums of its classes apart (more registers, 0 - 4 % of a batch's time: eight 24 x 20 x 20 x 1024
    // 83.8 -> 85.8 us, eight 32 x 16 x 16 x 1024 66.7 -> 67.4; with the narrow slices themselves 87.8 and
    // 71.7).
    if constexpr (V > 1) {
        const long long enough = 2LL * sm_count();
        const int nq16 = (p.C + 16 * V - 1) / (16 * V);
        auto width = [&](long long rows) { return rows * p.nq >= enough ? 32 : (rows * nq16 >= enough ? 16 : 8); };
        const int alone = width(p.F), here = width((long long)p.F * p.nclips);
        if (alone == 16) return here == 32 ? launch_sum_ls<T, V, 32, false, 2>(p, s, st) : launch_sum_ls<T, V, 16, false>(p, s, st);
        if (alone == 8)
            return here == 32 ? launch_sum_ls<T, V, 32, false, 4>(p, s, st)
                 : here == 16 ? launch_sum_ls<T, V, 16, false, 2>(p, s, st) : launch_sum_ls<T, V, 8, false>(p, s, st);
    }
    return launch_sum_ls<T, V, 32, false>(p, s, st);
}

// The query's counts of fused tokens start at zero for the matching kernel: cleared by the kernel between the sweep and it
// (all CTAs of the grid; a parameter more in the sweep cost it a CTA per SM in registers, 37.8 -> 39.5 us per pass).
__device__ __forceinline__ void clear_counts(int* fuse_cnt, int N) {
    if (!fuse_cnt) return;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) fuse_cnt[j] = 0;
}

// ---------------------------------------------------------------------------------------------------------
constexpr int kStatFB = 4;           // frames per thread held in registers (8 warps x 4 = 32 frames)

template <int V> __device__ __forceinline__ void load_f32(const float* p, float (&x)[V]);
template <> __device__ __forceinline__ void load_f32<4>(const float* p, float (&x)[4]) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(p));
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
}
template <> __device__ __forceinline__ void load_f32<1>(const float* p, float (&x)[1]) { x[0] = __ldcg(p); }

// A CTA owns a slice of kStatSub*32*V channels: warp = frame row (frames w, w+8, ...), lane = V channels in each
// of the kStatSub sub-slices.  V = 4 when C is a multiple of 4 (16-byte loads of the fp32 frame sums), else 1.
constexpr int kStatSub = 1;

template <int V>
__global__ void __launch_bounds__(kNormThreads)
k_frame_stats(const float* S, int F, int C, int nsl, float* Dp, float* Qp, float* Gp, int* hdr, int* out_anchor,
              size_t sstride, int* fuse_cnt, int N)
{
    S = clip_block(S, sstride); Dp = clip_block(Dp, sstride); Qp = clip_block(Qp, sstride); Gp = clip_block(Gp, sstride);
    hdr = clip_block(hdr, sstride);
    pdl_launch_dependents();
    trace_mark(hdr, 1, false);
    pdl_wait();                                      // the sweep's frame sums are complete and visible
    trace_mark(hdr, 4, false);
    clear_counts(fuse_cnt, N);
    const int q = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int NV = kStatSub * V;                 // channels per lane
    __shared__ float s_gp[kNormWarps][32 * NV];
    int c0[kStatSub];
    bool on[kStatSub];
#pragma unroll
    for (int sb = 0; sb < kStatSub; ++sb) {
        c0[sb] = ((q * kStatSub + sb) * 32 + lane) * V;
        on[sb] = c0[sb] < C;                         // C % V == 0
    }
    const bool resident = F <= kNormWarps * kStatFB; // this thread's frame sums all stay in registers

    auto load_frames = [&](int kb, float (&acc)[kStatFB][NV]) {
#pragma unroll
        for (int jj = 0; jj < kStatFB; ++jj) {
            const int kk = kb + jj * kNormWarps;
#pragma unroll
            for (int sb = 0; sb < kStatSub; ++sb) {
                float x[V];
                if (on[sb] && kk < F) load_f32<V>(S + (size_t)kk * C + c0[sb], x);
                else {
#pragma unroll
                    for (int v = 0; v < V; ++v) x[v] = 0.f;
                }
#pragma unroll
                for (int v = 0; v < V; ++v) acc[jj][sb * V + v] = x[v];
            }
        }
    };

    float acc[kStatFB][NV];
    float gacc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) gacc[v] = 0.f;
    for (int kb = w; kb < F; kb += kNormWarps * kStatFB) {
        load_frames(kb, acc);
#pragma unroll
        for (int jj = 0; jj < kStatFB; ++jj)
#pragma unroll
            for (int v = 0; v < NV; ++v) gacc[v] += acc[jj][v];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) s_gp[w][lane * NV + v] = gacc[v];
    __syncthreads();
    float gl[NV];                                    // g[c] = sum_k S_k[c], warps combined in warp order
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        float g = 0.f;
#pragma unroll
        for (int ww = 0; ww < kNormWarps; ++ww) g += s_gp[ww][lane * NV + v];
        gl[v] = g;
    }
    for (int kb = w; kb < F; kb += kNormWarps * kStatFB) {     // trip count is uniform inside a warp
        if (!resident) load_frames(kb, acc);
#pragma unroll
        for (int jj = 0; jj < kStatFB; ++jj) {
            const int kk = kb + jj * kNormWarps;
            float d = 0.f, qq = 0.f;
#pragma unroll
            for (int v = 0; v < NV; ++v) { d = fmaf(acc[jj][v], gl[v], d); qq = fmaf(acc[jj][v], acc[jj][v], qq); }
            d = warp_sum(d);
            qq = warp_sum(qq);
            if (lane < kStatReplicas && kk < F) {             // every lane holds the sums: one lane per replica
                Dp[((size_t)lane * nsl + q) * F + kk] = d;
                Qp[((size_t)lane * nsl + q) * F + kk] = qq;
            }
        }
    }
    if (w == 0) {
        float gg = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) gg = fmaf(gl[v], gl[v], gg);
        gg = warp_sum(gg);
        if (lane < kStatReplicas) Gp[(size_t)lane * nsl + q] = gg;
    }

    // The CTA that finishes last takes the arg max over the frames (Eq. auto_anchor) for the whole clip, so that the
    // CTAs of the matching kernel only read one word instead of each repeating the search while they hold most of an
    // SM.  The arrival counter is left at zero for the next call.
    __shared__ int s_last;
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(hdr + HDR_DONE_ALL, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        AnchorSrc src;
        src.Dp = Dp; src.Qp = Qp; src.Gp = Gp; src.nsl = nsl; src.fixed = -1; src.from_hdr = 0; src.hdr = hdr;
        src.out_anchor = out_anchor;
        const int a = resolve_anchor(src, F);
        if (tid == 0) {
            hdr[HDR_ANCHOR] = a;
            if (out_anchor) *out_anchor = a;
            hdr[HDR_DONE_ALL] = 0;
        }
    }
    trace_mark(hdr, 1, true);
}

// ---------------------------------------------------------------------------------------------------------
// The same statistics as ONE thread-block cluster of CS = 1, 8 or 16 CTAs, for clips of at most 4096 channels and 256
// frames (the frame sums of up to 128 / SL frames at SL slices of 128 channels per CTA stay in registers; longer clips
// are fetched a second time for the second step).  A grid of
// independent CTAs has to go through global memory, a fence and an arrival counter before one of them can take
// the arg max, which is five to six dependent round trips after the sweep; here every CTA fetches all of its
// frame sums in one round trip, the per-frame shares of <S_k, g>, |S_k|^2 and |g|^2 go to rank 0 through
// distributed shared memory, and rank 0 takes the arg max after one cluster barrier (7.2 -> 4.8 us per launch on
// the 8B-shaped clip, 42.1 -> 37.7 us per clip with one clip in flight).  Every order of summation is fixed and a function of
// the clip's shape: with more than eight slices the unit is one sixteenth of them (slices v, v + 16), two units v and v + 8
// are added first and these pairs in order, whether eight CTAs hold a pair each or sixteen a unit each.  (The grid kernel
// adds the same terms in an order of its own; which of the two a clip takes depends on its shape alone.)
// What bounds it is a serial chain: what an SM can take in from L2 (64 KB per CTA for 32 frames of 4096 channels on eight
// CTAs, 0.9 us; hence sixteen where the kernel runs alone), three block barriers and the cluster barrier.
// With eight CTAs, two shuffle trees per frame and every warp adding up all channels of g for itself a pass took, in a
// replayed graph, 39.3 us (32 x 16 x 16 x 4096), 28.9 (2048 channels), 134.7 (128 frames) and 11.3 (4 x 8 x 8 x 64) where it
// took 38.0, 28.1, 130.2 and 10.2, without the folds of frames that a clip does not have 0.3 - 0.4 less again; the order of summation that eight and sixteen CTAs share added nothing (39.8 -> 39.6 and
// 28.5 -> 28.3 per call).
constexpr int kStatClusterMaxF = 256;     // frames the cluster kernel takes (shares of all frames live in shared memory)

template <int SL, int CS>     // slices of 128 channels per CTA, CTAs; warp w owns frames w, w + 8, ...
__global__ void __launch_bounds__(kNormThreads)
k_frame_stats_cluster(const float* S, int F, int C, int nsl, int* hdr, int* out_anchor, size_t sstride, int* fuse_cnt, int N)
{
    S = clip_block(S, sstride); hdr = clip_block(hdr, sstride);
    constexpr int FB = 16 / SL;                      // frames per thread and chunk
    constexpr int CHUNK = kNormWarps * FB;           // frames per chunk: 32 / 64 / 128
    __shared__ float s_g[kNormWarps][SL * 128];
    __shared__ float s_gl[SL * 128];
    __shared__ float s_D[kStatClusterMaxF], s_Q[kStatClusterMaxF], s_G;
    __shared__ float s_x[CS > 1 ? CS - 1 : 1][2 * kStatClusterMaxF + 1];   // what the other ranks send (rank 0 only)
    __shared__ float s_best[kNormWarps];
    __shared__ int s_idx[kNormWarps];
    pdl_launch_dependents();
    if (CS > 1) cluster_arrive();                    // this CTA runs: the others may write into it
    trace_mark(hdr, 1, false);
    pdl_wait();                                      // the sweep's frame sums are complete and visible
    trace_mark(hdr, 4, false);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rank = CS > 1 ? (int)cluster_rank() : 0;
    const bool one_chunk = F <= CHUNK;               // then the frame sums stay in registers for the second step

    clear_counts(fuse_cnt, N);

    // the frame sums of one chunk of frames: one round trip
    float4 v[SL][FB];
    auto load_chunk = [&](int k0) {
#pragma unroll
        for (int sl = 0; sl < SL; ++sl) {
            const int q = rank + sl * CS;
            const int c0 = (q * 32 + lane) * 4;
#pragma unroll
            for (int jj = 0; jj < FB; ++jj) {
                const int kk = k0 + w + jj * kNormWarps;
                v[sl][jj] = (q < nsl && c0 < C && kk < F) ? __ldcg(reinterpret_cast<const float4*>(S + (size_t)kk * C + c0))
                                                          : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    // step 1: g[c] = sum_k S_k[c] over all frames (chunks in order, then the warps in warp order)
    float4 gacc[SL];
#pragma unroll
    for (int sl = 0; sl < SL; ++sl) gacc[sl] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < F; k0 += CHUNK) {
        load_chunk(k0);
#pragma unroll
        for (int sl = 0; sl < SL; ++sl)
#pragma unroll
            for (int jj = 0; jj < FB; ++jj) {
                gacc[sl].x += v[sl][jj].x; gacc[sl].y += v[sl][jj].y; gacc[sl].z += v[sl][jj].z; gacc[sl].w += v[sl][jj].w;
            }
    }
#pragma unroll
    for (int sl = 0; sl < SL; ++sl) reinterpret_cast<float4*>(s_g[w])[sl * 32 + lane] = gacc[sl];
    __syncthreads();
    for (int c = tid; c < SL * 128; c += kNormThreads) {          // one channel per thread
        float g = 0.f;
#pragma unroll
        for (int ww = 0; ww < kNormWarps; ++ww) g += s_g[ww][c];
        s_gl[c] = g;
    }
    __syncthreads();
    float4 gl[SL];
#pragma unroll
    for (int sl = 0; sl < SL; ++sl) gl[sl] = reinterpret_cast<const float4*>(s_gl)[sl * 32 + lane];
    // step 2: this CTA's shares of <S_k, g> and |S_k|^2 for every frame, eight sums at a time added up over the warp (fold8):
    // four frames, or two frames of two units (even and odd slices of this CTA), which are then added
    constexpr int U = CS == 8 && SL > 1 ? 2 : 1;     // units of this CTA
    constexpr int FP = 4 / U;                        // frames per fold
    // One CTA adds up each slice apart (2 or 4 of them, as a tree): small shares of one slice are not lost in a large one of another
    // while a chain runs through both.  (Root mean square error of the cosines against 64 bits, a numpy model of the three orders, in
    // units of 1e-8, a chain through the slices / apart / a CTA per slice: two slices 4.58 / 4.56 / 4.55, three 4.65 / 4.58 / 4.65,
    // four 4.62 / 4.52 / 4.90.)
    auto apart = [](const float (&x)[SL]) { return SL == 4 ? (x[0] + x[SL / 4]) + (x[SL / 2] + x[SL - 1]) : (SL == 2 ? x[0] + x[SL - 1] : x[0]); };
    for (int k0 = 0; k0 < F; k0 += CHUNK) {
        if (!one_chunk) load_chunk(k0);              // (a second round trip per chunk for clips of several chunks)
#pragma unroll
        for (int j0 = 0; j0 < FB; j0 += FP) {
            if (k0 + w + j0 * kNormWarps >= F) break;    // (no frames left for this warp: a fold is 450 cycles)
            float part[8];                           // [<S_k, g> or |S_k|^2][unit][frames j0 .. j0 + FP - 1]
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float d = 0.f, qq = 0.f, ds[SL], qs[SL];
#pragma unroll
                for (int sl = e / FP; sl < SL; sl += U) {
                    const float4 x = v[sl][j0 + e % FP], g = gl[sl];
                    if (CS == 1) d = qq = 0.f;
                    d = fmaf(x.x, g.x, d); d = fmaf(x.y, g.y, d); d = fmaf(x.z, g.z, d); d = fmaf(x.w, g.w, d);
                    qq = fmaf(x.x, x.x, qq); qq = fmaf(x.y, x.y, qq); qq = fmaf(x.z, x.z, qq); qq = fmaf(x.w, x.w, qq);
                    ds[sl] = d; qs[sl] = qq;
                }
                part[e] = CS == 1 ? apart(ds) : d; part[4 + e] = CS == 1 ? apart(qs) : qq;
            }
            float tot = fold8(part, lane);           // lanes 0, 4, 8, ..: part[4 * bit4 + 2 * bit3 + bit2] of the lane index
            if (U == 2) tot += __shfl_xor_sync(0xffffffffu, tot, 8);
            const int kk = k0 + w + (j0 + (U == 2 ? 0 : (lane >> 3) & 1) * 2 + ((lane >> 2) & 1)) * kNormWarps;
            if ((lane & (U == 2 ? 11 : 3)) == 0 && kk < F) (lane & 16 ? s_Q : s_D)[kk] = tot;
        }
    }
    if (w == 0) {
        float gg = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float part = 0.f, ps[SL];
#pragma unroll
            for (int sl = u; sl < SL; sl += U) {
                const float4 g = gl[sl];
                if (CS == 1) part = 0.f;
                part = fmaf(g.x, g.x, part); part = fmaf(g.y, g.y, part); part = fmaf(g.z, g.z, part); part = fmaf(g.w, g.w, part);
                ps[sl] = part;
            }
            part = warp_sum(CS == 1 ? apart(ps) : part);
            gg = u == 0 ? part : gg + part;
        }
        if (lane == 0) s_G = gg;
    }
    __syncthreads();
    if (CS > 1) {
        cluster_wait();                              // every CTA has started
        if (rank > 0) {                              // hand the shares to rank 0
            for (int i = tid; i < 2 * F + 1; i += kNormThreads)
                st_cluster_f32(cluster_addr(smem_u32(&s_x[rank - 1][i]), 0),
                               i < F ? s_D[i] : (i < 2 * F ? s_Q[i - F] : s_G));
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    }
    if (rank == 0) {
        // Eq. (auto_anchor): a* = arg max_k <S_k, g> / (|S_k| |g|), lowest frame on ties; ranks added in order
        float best = -INFINITY;
        int idx = 0x7fffffff;
        if (tid < F) {                               // F <= kStatClusterMaxF = the CTA's 256 threads
            // what rank r holds, and with sixteen ranks what rank r + 8 holds added to it first
            auto share = [&](int r, int i, float own) {
                const float x = r == 0 ? own : s_x[r - 1][i];
                return CS == 16 ? x + s_x[CS == 16 ? r + 7 : 0][i] : x;
            };
            float D = share(0, tid, s_D[tid]), Q = share(0, F + tid, s_Q[tid]), G = share(0, 2 * F, s_G);
#pragma unroll
            for (int r = 1; r < (CS < 8 ? CS : 8); ++r) {
                D += share(r, tid, 0.f); Q += share(r, F + tid, 0.f); G += share(r, 2 * F, 0.f);
            }
            best = D * (1.0f / fmaxf(sqrtf(G), kNormFloor)) * (1.0f / fmaxf(sqrtf(Q), kNormFloor));
            idx = tid;
        }
        auto better = [](float ob, int oi, float& best, int& idx) {
            const bool take = (oi != 0x7fffffff) & ((idx == 0x7fffffff) | (ob > best) | ((ob == best) & (oi < idx)));
            best = take ? ob : best;
            idx = take ? oi : idx;
        };
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
            better(ob, oi, best, idx);
        }
        if (F > 32) {
            if (lane == 0) { s_best[w] = best; s_idx[w] = idx; }
            __syncthreads();
            if (tid == 0)
                for (int ww = 1; ww < kNormWarps; ++ww) better(s_best[ww], s_idx[ww], best, idx);
        }
        if (tid == 0) {
            hdr[HDR_ANCHOR] = idx;
            if (out_anchor) *out_anchor = idx;
        }
    }
    trace_mark(hdr, 1, true);
}

// clusters of sixteen CTAs: allowed for `func` on the current device (set once)
static cudaError_t ensure_large_clusters(const void* func) {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count({func, dev})) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) done.insert({func, dev});
    return e;
}

template <int SL, int CS>
static cudaError_t launch_stats_cluster_t(const Problem& p, const Scratch& s, int* out_anchor, cudaStream_t st) {
    const auto kernel = k_frame_stats_cluster<SL, CS>;
    if (CS > 8) {                                    // (sixteen CTAs to a cluster have to be asked for)
        cudaError_t e = ensure_large_clusters(reinterpret_cast<const void*>(kernel));
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS, p.nclips); cfg.blockDim = dim3(kNormThreads); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = CS > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, (const float*)s.S, p.F, p.C, p.nsl, s.hdr, out_anchor, p.sstride,
                              p.fuse_cnt, p.N);
}

// What the sweep leaves behind besides its sums, for calls that need no sweep (a fixed anchor and a matching kernel
// that takes the token norms itself): survivor counters at zero, error word cleared.
__global__ void __launch_bounds__(256)
k_begin_call(int F, int* __restrict__ cnt, int* __restrict__ hdr, size_t sstride, int* fuse_cnt, int N, int fresh)
{
    cnt = clip_block(cnt, sstride); hdr = clip_block(hdr, sstride);
    pdl_launch_dependents();
    pdl_wait();                                      // the previous call's gather may still read the counters
    for (int k = threadIdx.x; k < F; k += 256) cnt[k] = 0;
    clear_counts(fuse_cnt, N);
    if (threadIdx.x == 0) clear_words(hdr, fresh);
}

cudaError_t launch_norm_sum(const Problem& p, const Scratch& s, cudaStream_t st) {
    if (p.anchor_mode != 0 && !needs_sweep_norms(p))           // Eq. (auto_anchor) is not evaluated: no pass over X
        return launch_ex(true, 0, k_begin_call, dim3(1, p.nclips), dim3(256), st, p.F, s.cnt, s.hdr, p.sstride,
                         p.fuse_cnt, p.N, p.fresh);
    if (p.dtype == 0) return p.vec ? launch_sum_t<float, 4>(p, s, st) : launch_sum_t<float, 1>(p, s, st);
    return p.vec ? launch_sum_t<bf16_t, 8>(p, s, st) : launch_sum_t<bf16_t, 1>(p, s, st);
}

// whether the current device can run such a cluster of the statistics kernel (asked once per device)
static bool large_clusters() {
    static std::mutex mu;
    static std::map<int, bool> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(dev);
    if (it != known.end()) return it->second;
    const auto kernel = k_frame_stats_cluster<2, 16>;
    int n = 0;
    if (ensure_large_clusters(reinterpret_cast<const void*>(kernel)) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16); cfg.blockDim = dim3(kNormThreads);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 16; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
        cfg.attrs = &attr; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = 0;
    }
    return known[dev] = n > 0;
}

cudaError_t launch_frame_stats(const Problem& p, const Scratch& s, int* out_anchor, cudaStream_t st) {
    if (p.anchor_mode != 0) return cudaSuccess;                // fixed anchors need no statistics
    // The single-cluster kernel is the shorter one (4.9 against 7.2 us on a 32-frame clip of 4096 channels) and takes
    // every clip it can.  Sixteen CTAs where nothing runs beside the call, eight in a batch: a cluster starts only when all
    // its places in one GPC are free at the same moment.
    if (p.C % 4 == 0 && p.nsl <= 32 && p.F <= kStatClusterMaxF) {
        if (p.nsl == 1) return launch_stats_cluster_t<1, 1>(p, s, out_anchor, st);      // nothing to split
        // Two to four slices of so few frames that one CTA holds their sums (64 KB) at once: what the other CTAs would save is
        // less than the exchange between them costs (1200 cycles; us per pass with eight CTAs / one: 24 x 20 x 15 x 248
        // 15.5 / 14.9, 16 x 14 x 14 x 512 13.2 / 12.8, 32 x 14 x 14 x 512 14.4 / 14.2, 52 x 14 x 9 x 208 14.0 / 13.6; eight
        // slices, 16 x 16 x 16 x 1024 15.2 / 15.4).
        if (p.nsl == 2 && p.F <= 64) return launch_stats_cluster_t<2, 1>(p, s, out_anchor, st);
        if (p.nsl <= 4 && p.F <= 32) return launch_stats_cluster_t<4, 1>(p, s, out_anchor, st);
        const bool alone = p.overlapped <= 1 && large_clusters();
        if (p.nsl > 16) return alone ? launch_stats_cluster_t<2, 16>(p, s, out_anchor, st)
                                     : launch_stats_cluster_t<4, 8>(p, s, out_anchor, st);
        if (p.nsl > 8) return alone ? launch_stats_cluster_t<1, 16>(p, s, out_anchor, st)
                                    : launch_stats_cluster_t<2, 8>(p, s, out_anchor, st);
        return launch_stats_cluster_t<1, 8>(p, s, out_anchor, st);
    }
    if (p.C % 4 == 0)
        return launch_pdl(k_frame_stats<4>, dim3(p.nsl, p.nclips), dim3(kNormThreads), st, (const float*)s.S, p.F, p.C, p.nsl,
                          s.Dp, s.Qp, s.Gp, s.hdr, out_anchor, p.sstride, p.fuse_cnt, p.N);
    return launch_pdl(k_frame_stats<1>, dim3(p.nsl, p.nclips), dim3(kNormThreads), st, (const float*)s.S, p.F, p.C, p.nsl,
                      s.Dp, s.Qp, s.Gp, s.hdr, out_anchor, p.sstride, p.fuse_cnt, p.N);
}

}  // namespace ttf
