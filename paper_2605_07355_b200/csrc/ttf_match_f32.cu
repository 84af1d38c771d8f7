// Pointwise Matching with Local Window Search and Threshold Gating (Eqs. pi, argmax, dst, gating, mask) for fp32 clips
// with 16-byte aligned rows and r <= 2, on the fp32 pipes.
//
// A CTA owns one grid cell and FR frames of it: FR source rows against the (2r+1)^2 anchor rows around the cell.
// Stages of kF32KC channels arrive as two TMA tensor tiles (the source rows; the window rows, zero-filled outside the
// grid) in an mbarrier ring; a warp owns FW of the frames, a lane owns 4 channels of every 128, and keeps all FW x WIN
// dot products and the FW + WIN squared norms of its rows as running sums in registers, so that a window row read from
// shared memory serves FW source rows and a source row WIN candidates.  The lanes are added up once, at the end.
//
// What bounds it: shared memory (FW + WIN rows of 512 bytes are read per FW x WIN x 4 multiply-adds of a lane) and the
// fp32 pipes are within a few per cent of each other at r = 1 (68 against 89 cycles of an SM per warp and stage), and
// both stay below what an SM takes in from L2 (FR + WIN rows per stage).  The CUDA-core kernel that it
// replaced here gave a warp one token and read every window row again for every token: on a 32 x 16 x 16 clip of 1152
// channels 67 us of a pass of 81.8 us; the pass takes 30.3 us now (no norms in the sweep either).
#include <cuda.h>

#include "ttf_internal.cuh"
#include "ttf_async.cuh"
#include "ttf_tensormap.cuh"

namespace ttf {

constexpr int kF32KC = 128;              // channels per stage: one 16-byte piece per lane
constexpr int kF32Row = kF32KC * 4;      // bytes of a row of a stage

template <int R> struct F32Shape {
    static constexpr int SIDE = 2 * R + 1;
    static constexpr int WIN = SIDE * SIDE;
    static constexpr int FW = R == 2 ? 4 : 8;             // frames per warp (registers: FW * WIN + FW + WIN sums)
    static constexpr int MAXW = 32 / FW;                  // warps of the largest CTA: 32 frames
    static constexpr int STAGES = R == 2 ? 3 : 4;         // two CTAs of 32 frames per SM
    static constexpr int NV = FW * WIN + FW + WIN;        // sums per lane
    static constexpr int NG = (NV + 31) / 32;             // ... in groups of 32 for the reduction over the lanes
};

// Sum of v[i] over the warp for i = 0..31 with 31 shuffles; lane l returns the total of v[l].
__device__ __forceinline__ float fold32(float (&v)[32], int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? v[i] : v[i + o];
            const float keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

template <int R, int G, int ST>      // ST: stages of the ring
__global__ void __launch_bounds__(F32Shape<R>::MAXW * 32)
k_match_f32(const __grid_constant__ ClipMaps<G> maps, int F, int H, int W, int C, float t, AnchorSrc asrc,
            float* __restrict__ shat, int* __restrict__ dst, unsigned char* __restrict__ keep, int* __restrict__ cnt,
            int wait_limit, int tx_extra, size_t sstride, int* fuse_cnt)
{
    const CUtensorMap& mapA = maps.a[blockIdx.y];
    const CUtensorMap& mapB = maps.b[blockIdx.y];
    asrc = clip_block(asrc, sstride); cnt = clip_block(cnt, sstride);
    shat = clip_block(shat, sstride); dst = clip_block(dst, sstride); keep = clip_block(keep, sstride);
    using S = F32Shape<R>;
    extern __shared__ __align__(128) unsigned char f32_ring[];
    __shared__ uint64_t bar[ST];
    __shared__ float s_sum[S::MAXW][S::NG * 32];
    __shared__ int s_err;
    const int N = H * W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int FR = (int)(blockDim.x >> 5) * S::FW;         // frames of this CTA
    const int i = blockIdx.x % N, k0 = (blockIdx.x / N) * FR;
    const int y = i / W, x = i - y * W;
    const int nst = (C + kF32KC - 1) / kF32KC;
    const uint32_t abytes = (uint32_t)FR * kF32Row, stage_bytes = abytes + S::WIN * kF32Row;

    trace_mark(asrc.hdr, 2, false);
    if (tid == 0) {
        for (int s = 0; s < ST; ++s) mbar_init(&bar[s], 1);
        mbar_init_fence();
        s_err = 0;
        tensormap_prefetch(&mapA);
        tensormap_prefetch(&mapB);
    }
    __syncthreads();
    pdl_wait();                                            // the anchor, and whatever produced X, is complete
    trace_mark(asrc.hdr, 5, false);
    const int a = asrc.fixed >= 0 ? asrc.fixed : __ldcg(asrc.hdr + HDR_ANCHOR);
    if (blockIdx.x == 0 && tid == 0 && asrc.fixed >= 0) {
        if (asrc.begins) clear_words(asrc.hdr, false);
        asrc.hdr[HDR_ANCHOR] = a;                          // the gather reads it from here
        if (asrc.out_anchor) *asrc.out_anchor = a;
    }

    auto issue = [&](int it, int slot) {                   // thread 0: both tiles of stage it
        unsigned char* s = f32_ring + (size_t)slot * stage_bytes;
        mbar_arrive_expect_tx(&bar[slot], stage_bytes + (uint32_t)tx_extra);      // (extra: test hook only)
        tma_load_4d(s, &mapA, it * kF32KC, x, y, k0, &bar[slot]);
        tma_load_4d(s + abytes, &mapB, it * kF32KC, x - R, y - R, a, &bar[slot]);
    };
    int issued = 0;
    if (tid == 0)
        for (; issued < ST && issued < nst; ++issued) issue(issued, issued);

    float acc[S::FW][S::WIN], na[S::FW], nb[S::WIN];
#pragma unroll
    for (int f = 0; f < S::FW; ++f) {
        na[f] = 0.f;
#pragma unroll
        for (int c = 0; c < S::WIN; ++c) acc[f][c] = 0.f;
    }
#pragma unroll
    for (int c = 0; c < S::WIN; ++c) nb[c] = 0.f;

    bool ok = true;                                        // (per thread: a thread whose wait ran out stops computing,
    int slot = 0;                                          // but takes part in every barrier)
    uint32_t parity = 0;
    for (int it = 0; it < nst; ++it) {
        if (ok && !mbar_wait(&bar[slot], parity, wait_limit)) { ok = false; atomicExch(&s_err, 1); }
        if (ok) {
            const unsigned char* sa = f32_ring + (size_t)slot * stage_bytes + lane * 16;
            const float4* ra = reinterpret_cast<const float4*>(sa + (size_t)w * S::FW * kF32Row);
            const float4* rb = reinterpret_cast<const float4*>(sa + abytes);
            float4 va[S::FW];
#pragma unroll
            for (int f = 0; f < S::FW; ++f) va[f] = ra[f * (kF32Row / 16)];
#pragma unroll
            for (int f = 0; f < S::FW; ++f) na[f] = dot4(va[f], va[f], na[f]);
#pragma unroll
            for (int c = 0; c < S::WIN; ++c) {
                const float4 vb = rb[c * (kF32Row / 16)];
                nb[c] = dot4(vb, vb, nb[c]);
#pragma unroll
                for (int f = 0; f < S::FW; ++f) acc[f][c] = dot4(va[f], vb, acc[f][c]);
            }
        }
        if (it + ST < nst) {                               // the stage is free: refill it
            __syncthreads();
            if (tid == 0 && !*(volatile int*)&s_err) { issue(it + ST, slot); issued = it + ST + 1; }
        }
        if (++slot == ST) { slot = 0; parity ^= 1; }
    }
    if (tid == 0 && *(volatile int*)&s_err) {
        // copies still land in this CTA's shared memory: wait (bounded again) for the stages issued last
        for (int it = issued > ST ? issued - ST : 0; it < issued; ++it)
            mbar_wait(&bar[it % ST], (it / ST) & 1, wait_limit);
        report_give_up(asrc.hdr, asrc.begins);
    }
    pdl_launch_dependents();                               // (not at the start: the gather's CTAs would take the place
                                                           // of other clips' kernels while this one runs)
    // one value per (frame, candidate), per frame and per candidate: added up over the lanes, 32 values at a time
#pragma unroll
    for (int g = 0; g < S::NG; ++g) {
        float v[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const int q = g * 32 + e;
            v[e] = q < S::FW * S::WIN ? acc[q / S::WIN < S::FW ? q / S::WIN : 0][q % S::WIN]
                 : q < S::FW * S::WIN + S::FW ? na[q - S::FW * S::WIN < S::FW ? q - S::FW * S::WIN : 0]
                 : q < S::NV ? nb[q - S::FW * S::WIN - S::FW < S::WIN ? q - S::FW * S::WIN - S::FW : 0] : 0.f;
        }
        s_sum[w][g * 32 + lane] = fold32(v, lane);
    }
    __syncwarp();
    float* sum = s_sum[w];
    if (lane < S::FW + S::WIN) {                           // 1 / max(||x||, floor) of the source and the window rows
        float& n2 = sum[S::FW * S::WIN + lane];
        n2 = 1.0f / fmaxf(sqrtf(n2), kNormFloor);
    }
    static_assert(S::FW + S::WIN <= 32, "one lane per norm");
    __syncwarp();
    const int k = k0 + w * S::FW + lane;
    if (lane < S::FW && k < F && in_bounds(asrc.hdr, 2, (long long)k * N + i, (long long)F * N)) {
        const size_t f = (size_t)k * N + i;
        if (k == a) {                                      // anchor tokens are always retained (Eq. mask)
            shat[f] = 1.0f; dst[f] = i; keep[f] = 1;
        } else {
            const float rs = sum[S::FW * S::WIN + lane];
            float best = -INFINITY;
            int best_j = -1;
#pragma unroll
            for (int c = 0; c < S::WIN; ++c) {             // ascending anchor index among in-grid cells
                const int yy = y + c / S::SIDE - R, xx = x + c % S::SIDE - R;
                if (yy < 0 || yy >= H || xx < 0 || xx >= W) continue;
                const float sim = sum[lane * S::WIN + c] * rs * sum[S::FW * S::WIN + S::FW + c];
                if (sim > best || best_j < 0) { best = sim; best_j = yy * W + xx; }
            }
            gate_token(best, best_j, t, f, shat, dst, keep, cnt + k, fuse_cnt);
        }
    }
    trace_mark(asrc.hdr, 2, true);
}

// Stages of the ring.  At r <= 1 a ring of four leaves room for two CTAs of 32 frames on an SM, one of three for three,
// which is better where a launch then fits the GPU at once, or is several times what fits.  (At r = 2 the registers leave
// room for one CTA of 32 frames whatever its ring.)  No more than the channels fill, so that short rows make room for more
// CTAs.  A launch that fits with the whole ring keeps it (us per pass, replayed graph, whole ring / as here: 98 x 10 x 32 x
// 352 37.1 / 32.5, 64 x 24 x 24 x 512 46.4 / 43.9, two of 102 x 15 x 12 x 288 40.0 / 37.7 and, measured again, 39.0 / 38.4,
// 34 x 15 x 15 x 3312 at r = 0 68.3 / 62.7; with three stages where this takes four, 68 x 13 x 15 x 2520 84.7 / 95.0 and 32
// x 16 x 16 x 1152 22.7 / 24.4).
template <int R> static int ring_stages(const Problem& p, long long units, int FR) {
    using S = F32Shape<R>;
    const int nst = (p.C + kF32KC - 1) / kF32KC;
    auto places = [&](int stages) { return (long long)sm_count() * (220 * 1024 / (stages * (FR + S::WIN) * kF32Row)); };
    if (units <= places(S::STAGES)) return S::STAGES;
    if (nst < S::STAGES) return nst < 2 ? 2 : nst;
    return R < 2 && (units <= places(3) || units > 2 * places(3)) ? 3 : S::STAGES;
}

template <int R, int G, int ST>
static cudaError_t launch_f32_ring(const Problem& p, const Scratch& s, const ClipMaps<G>& maps, int FR, unsigned units, int* out_anchor,
                                   float* shat, int* dst, unsigned char* keep, cudaStream_t st) {
    using S = F32Shape<R>;
    const auto kernel = k_match_f32<R, G, ST>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (size_t)ST * (32 + S::WIN) * kF32Row);
    if (e != cudaSuccess) return e;
    return launch_ex(true, (size_t)ST * (FR + S::WIN) * kF32Row, kernel, dim3(units, p.nclips), dim3(FR / S::FW * 32), st, maps, p.F, p.H,
                     p.W, p.C, p.t, make_anchor_src(p, s, out_anchor), shat, dst, keep, s.cnt, wait_poll_limit(), wait_tx_extra(),
                     p.sstride, p.fuse_cnt);
}

// Frames per CTA: 32 reads the window rows least often (41 rows per 32 at r = 1, 25 per 16), but a grid of fewer than
// three CTAs per two SMs leaves SMs idle: then 16, then 8 (at least FW).
template <int R, int G>
static cudaError_t launch_f32_t(const Problem& p, const Scratch& s, int* out_anchor, float* shat, int* dst,
                                unsigned char* keep, cudaStream_t st) {
    using S = F32Shape<R>;
    int FR = 32;
    while (FR > S::FW && (FR / 2 >= p.F || (long long)p.N * p.nclips * ((p.F + FR - 1) / FR) * 2 < 3LL * sm_count())) FR /= 2;
    ClipMaps<G> maps;
    for (int n = 0; n < p.nclips; ++n)
        if (!make_tensor_map(&maps.a[n], p.xs.X[n], 0, p.F, p.H, p.W, p.C, kF32KC, 1, 1, FR, false) ||
            !make_tensor_map(&maps.b[n], p.xs.X[n], 0, p.F, p.H, p.W, p.C, kF32KC, S::SIDE, S::SIDE, 1, false))
            return cudaErrorInvalidValue;
    const long long units = (long long)p.N * ((p.F + FR - 1) / FR);
    const int stages = ring_stages<R>(p, units * p.nclips, FR);
    if constexpr (R < 2)
        if (stages == 4) return launch_f32_ring<R, G, 4>(p, s, maps, FR, (unsigned)units, out_anchor, shat, dst, keep, st);
    return stages == 3 ? launch_f32_ring<R, G, 3>(p, s, maps, FR, (unsigned)units, out_anchor, shat, dst, keep, st)
                       : launch_f32_ring<R, G, 2>(p, s, maps, FR, (unsigned)units, out_anchor, shat, dst, keep, st);
}

cudaError_t launch_match_f32(const Problem& p, const Scratch& s, int* out_anchor, float* shat, int* dst,
                             unsigned char* keep, cudaStream_t st) {
    if (p.nclips > 1) {
        if (p.r == 0) return launch_f32_t<0, kMaxGroup>(p, s, out_anchor, shat, dst, keep, st);
        if (p.r == 1) return launch_f32_t<1, kMaxGroup>(p, s, out_anchor, shat, dst, keep, st);
        return launch_f32_t<2, kMaxGroup>(p, s, out_anchor, shat, dst, keep, st);
    }
    if (p.r == 0) return launch_f32_t<0, 1>(p, s, out_anchor, shat, dst, keep, st);
    if (p.r == 1) return launch_f32_t<1, 1>(p, s, out_anchor, shat, dst, keep, st);
    return launch_f32_t<2, 1>(p, s, out_anchor, shat, dst, keep, st);
}

}  // namespace ttf
