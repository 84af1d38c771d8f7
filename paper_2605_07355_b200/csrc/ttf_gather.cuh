// Rank/select helpers of the output-driven gather kernels.
#pragma once

#include "ttf_internal.cuh"

namespace ttf {

constexpr int kCopyWarps = 8;
constexpr int kScanChunks = 4;       // frame counts per lane fetched at once by the warp-level frame search

// Exclusive prefix of the survivor counts of all frames in shared memory, for clips of up to kWarpPrefixMaxF frames
// (`pref`: [kWarpPrefixMaxF + 4]; pref[F] is the total, which is returned).  The anchor frame counts `acnt` tokens.  By all
// threads of a CTA of NW warps.  (Not for the gather with one row per warp at a time: its warps do better without a barrier
// before their first copy, 37.8 against 38.7 us per pass on 32 x 16 x 16 x 4096, 247 against 255 on 64 x 32 x 32 x 4096.)
template <int NW>
__device__ __forceinline__ int frame_prefix_cta(const int* cnt, int F, int a, int acnt, int* pref, int* s_warp) {
    static_assert(kWarpPrefixMaxF <= 4 * NW * 32, "four frames per thread");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, k = tid * 4;
    // (the counts are 256-byte aligned and followed by other scratch: a load that starts inside may run past their end)
    int4 v = k < F ? __ldcg(reinterpret_cast<const int4*>(cnt + k)) : make_int4(0, 0, 0, 0);
    int c[4] = {v.x, v.y, v.z, v.w};
    int mine = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        c[e] = k + e >= F ? 0 : (k + e == a ? acnt : c[e]);
        mine += c[e];
    }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    int at = incl - mine, total = 0;
#pragma unroll
    for (int ww = 0; ww < NW; ++ww) { at += ww < w ? s_warp[ww] : 0; total += s_warp[ww]; }
    if (k <= F && k < kWarpPrefixMaxF) {
#pragma unroll
        for (int e = 0; e < 4; ++e) { pref[k + e] = at; at += c[e]; }
    }
    if (F == kWarpPrefixMaxF && tid == 0) pref[F] = total;
    __syncthreads();
    return total;
}

// Frame that holds the e-th token of the walk (e < pref[F]).
__device__ __forceinline__ int frame_of(const int* pref, int F, int e) {
    int lo = 0, hi = F;                              // pref[lo] <= e < pref[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        const bool up = pref[mid] <= e;
        lo = up ? mid : lo;
        hi = up ? hi : mid;
    }
    return lo;
}

// Frame search of the gather: the frame that holds the e-th token of the flat walk and the number of walked tokens
// before that frame.  The walk visits the preserved tokens of the source frames in flat order; the anchor frame
// contributes `acnt` tokens: 0 when its rows are emitted as a block of their own (Eq. xprime_stack), N in natural
// order (all of its tokens are retained, Eq. mask).  Returns the total; k_out = -1 when e is past the end (e < 0
// asks for the total only).  All lanes of a warp call it with the same arguments.
__device__ __forceinline__ int find_frame(const int* __restrict__ cnt, const int* __restrict__ gprefix, int F, int a,
                                          int acnt, int lane, int e, int& k_out, int& before) {
    int running = 0;
    k_out = -1; before = 0;
    if (F > kWarpPrefixMaxF) {                         // pre-scanned prefix: binary search
        int lo = 0, hi = F;
        const int P = __ldcg(gprefix + F);
        if (e < P) {
            while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (__ldcg(gprefix + mid) <= e) lo = mid; else hi = mid; }
            k_out = lo; before = __ldcg(gprefix + lo);
        }
        return P;
    }
    for (int base = 0; base < F; base += 32 * kScanChunks) {
        int c[kScanChunks];
#pragma unroll
        for (int q = 0; q < kScanChunks; ++q) {
            const int k = base + q * 32 + lane;
            c[q] = k < F ? __ldcg(cnt + k) : 0;            // (unconditional: the load need not wait for the anchor word)
        }
#pragma unroll
        for (int q = 0; q < kScanChunks; ++q)
            if (base + q * 32 + lane == a) c[q] = acnt;
#pragma unroll
        for (int q = 0; q < kScanChunks; ++q) {
            int incl = c[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            if (k_out < 0 && e < running + total) {
                const unsigned m = __ballot_sync(0xffffffffu, running + incl > e);
                const int l = __ffs(m) - 1;
                k_out = base + q * 32 + l;
                before = running + __shfl_sync(0xffffffffu, incl - c[q], l);
            }
            running += total;
        }
        if (k_out >= 0 && e >= 0) break;               // e < 0 asks for the total only
    }
    return running;
}


// Cell index of the n-th (0-based) retained token of one frame: a warp-wide rank/select over the keep flags.
// All lanes must call with the same arguments; returns -1 if the frame holds fewer than n+1 retained tokens.
__device__ __forceinline__ int select_in_frame(const unsigned char* __restrict__ kf, int N, int n, int lane) {
    for (int b = 0; b < N; b += 256) {                     // 8 cells per lane, 256 per step
        const int c0 = b + lane * 8;
        unsigned bits = 0;
        if (c0 + 8 <= N && ((reinterpret_cast<uintptr_t>(kf + c0) & 7) == 0)) {
            const uint2 v = __ldcg(reinterpret_cast<const uint2*>(kf + c0));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                bits |= ((v.x >> (8 * e)) & 0xffu) ? (1u << e) : 0u;
                bits |= ((v.y >> (8 * e)) & 0xffu) ? (1u << (4 + e)) : 0u;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) bits |= (c0 + e < N && __ldcg(kf + c0 + e) != 0) ? (1u << e) : 0u;
        }
        const int mine = __popc(bits);
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (n < total) {
            const int excl = incl - mine;
            const bool here = n >= excl && n < incl;       // exactly one lane
            const int cell = here ? c0 + (int)__fns(bits, 0, n - excl + 1) : 0;
            const unsigned who = __ballot_sync(0xffffffffu, here);
            return __shfl_sync(0xffffffffu, cell, __ffs(who) - 1);
        }
        n -= total;
    }
    return -1;
}

}  // namespace ttf
