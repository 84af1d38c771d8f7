// Token Compression and Positional Alignment (Eqs. xprime_stack, mask, compress_pos, Lpre).
//
// The output position of a preserved source token is N plus the number of preserved source tokens before it
// in flat (k, i) order.  That exclusive prefix is taken in two levels: the per-frame survivor counts written
// by the matching kernel are scanned by every warp for itself (shuffles; a pre-scanned array for very long
// clips), and inside a frame the rank is a population count over the frame's keep flags.  The gather is then
// driven from the OUTPUT side: one warp per output row finds the source row by rank/select and copies it
// with all of its 16-byte loads in flight at once, so the work per warp is the same no matter how unevenly
// the survivors are spread over the frames.  No warp ever waits for another one.
#include "ttf_internal.cuh"
#include "ttf_async.cuh"
#include "ttf_gather.cuh"

#include <algorithm>

namespace ttf {

// exclusive scan of the effective per-frame counts (anchor frame counts as 0) for clips with more frames
// than fit the shared-memory scan of the gather kernel
__global__ void __launch_bounds__(1024)
k_frame_prefix(const int* __restrict__ cnt, const int* __restrict__ hdr, int F, int acnt, int* __restrict__ prefix,
               size_t sstride)
{
    cnt = clip_block(cnt, sstride); hdr = clip_block(hdr, sstride); prefix = clip_block(prefix, sstride);
    __shared__ int s_warp[32];
    __shared__ int s_carry;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int a = hdr[HDR_ANCHOR];
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < F; base += 1024) {
        const int k = base + tid;
        int v = k < F ? (k == a ? acnt : cnt[k]) : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int n = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += n;
        }
        if (lane == 31) s_warp[w] = incl;
        __syncthreads();
        if (w == 0) {
            int x = s_warp[lane], xi = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int n = __shfl_up_sync(0xffffffffu, xi, o);
                if (lane >= o) xi += n;
            }
            s_warp[lane] = xi - x;       // exclusive over warps
        }
        __syncthreads();
        const int carry = s_carry;
        if (k < F) prefix[k] = carry + s_warp[w] + incl - v;
        __syncthreads();
        if (tid == 1023) s_carry = carry + s_warp[w] + incl;
        __syncthreads();
    }
    if (tid == 0) prefix[F] = s_carry;
}

// COPY_BYTES: 16 when rows are 16-byte aligned multiples of 16 bytes, else the element size (2 or 4)
template <int COPY_BYTES> struct CopyUnit;
template <> struct CopyUnit<16> { using type = uint4; };
template <> struct CopyUnit<4> { using type = uint32_t; };
template <> struct CopyUnit<2> { using type = uint16_t; };

constexpr int kCopyUnroll = 8;       // 16-byte units in flight per lane of the element-wise gather (two steps for an 8 KB row)

// Gather with bulk asynchronous copies, for rows that are 16-byte aligned multiples of 16 bytes: a warp finds the
// source row of its output row by rank/select (frame search over the survivor counts, then a select inside that
// frame's keep flags), then one lane moves the row global -> shared -> global with two bulk copies per piece of at
// most kBulkPiece bytes, so no data passes through registers.  One row per warp at a time and 24 warps per SM:
// measured against variants in which a warp owns a contiguous range of rows, finds it with fewer dependent loads
// and keeps two to four rows in flight through a ring of slots, this plain form was the fastest (11.7 against
// 14.9 - 16.5 us on the 8B-shaped clip): the copies of a clip are one short burst that is bounded by what an SM can
// take in and put out per cycle, and what counts is how early the first copy of every warp is on its way.
// Every wait is bounded; a warp whose wait runs out stops copying, raises the error word and writes L' = -1.
constexpr int kBulkPiece = 8192;     // bytes per staging slot; longer rows go in pieces

__global__ void __launch_bounds__(kCopyWarps * 32)
k_compact_bulk(const __grid_constant__ ClipPtrs xs, size_t row_bytes, int F, int H, int W,
               int* __restrict__ hdr, const int* __restrict__ cnt, const int* __restrict__ gprefix,
               const unsigned char* __restrict__ keep, const __grid_constant__ OutPtrs outs, int NA, int acnt, int t_off, int pos_base,
               int late_trigger, int wait_limit, int tx_extra, int stream_once, size_t sstride)
{
    const unsigned char* __restrict__ X = reinterpret_cast<const unsigned char*>(xs.X[blockIdx.y]);
    unsigned char* __restrict__ out_tokens = reinterpret_cast<unsigned char*>(outs.tokens[blockIdx.y]);
    int* __restrict__ out_pos = outs.pos[blockIdx.y];
    int* __restrict__ out_count = outs.count[blockIdx.y];
    hdr = clip_block(hdr, sstride); cnt = clip_block(cnt, sstride); gprefix = clip_block(gprefix, sstride);
    keep = clip_block(keep, sstride);
    extern __shared__ __align__(128) unsigned char stage[];     // [kCopyWarps][kBulkPiece]
    __shared__ uint64_t bar[kCopyWarps];
    const int N = H * W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // The next kernel of the stream may be scheduled once every CTA has said so (or has exited).  Normally that is
    // said at once: the next kernel waits for this grid before it touches anything, and meanwhile its CTAs are set
    // up.  When the next kernel is the sweep of the next clip of a batch, which runs beside this gather without
    // waiting, it is said only after the wait below: the sweep must not start while the matching kernel still
    // needs this clip in L2.
    if (!late_trigger) pdl_launch_dependents();
    trace_mark(hdr, 3, false);
    if (lane == 0) { mbar_init(&bar[w], 1); mbar_init_fence(); }
    __syncwarp();
    pdl_wait();                                  // keep flags, dst and survivor counts are complete
    if (late_trigger) pdl_launch_dependents();
    trace_mark(hdr, 6, false);
    const int a = __ldcg(hdr + HDR_ANCHOR);
    const int gw = blockIdx.x * kCopyWarps + w;
    const int nw = gridDim.x * kCopyWarps;
    int Lp = 0;
    if (gw == 0) {                               // L' = N + P (Eq. Lpre)
        int kk, bb;
        Lp = NA + find_frame(cnt, gprefix, F, a, acnt, lane, -1, kk, bb);
        if (lane == 0) *reinterpret_cast<volatile int*>(out_count) = Lp;
    }
    unsigned char* buf = stage + (size_t)w * kBulkPiece;
    const int pieces = (int)((row_bytes + kBulkPiece - 1) / kBulkPiece);
    uint32_t phase = 0;
    bool gave_up = false;
    // the rows read here are not needed in L2 again, while the clip that is being matched and the one streaming in are: their
    // lines are the first to go; those of the rows written, which the caller reads next, only where they would not stay anyway
    const unsigned long long once = l2_evict_first_policy();
    for (int j = gw; ; j += nw) {
        int f;
        if (j < NA) f = a * N + j;               // anchor rows first (Eq. xprime_stack)
        else {
            int k, before;
            find_frame(cnt, gprefix, F, a, acnt, lane, j - NA, k, before);
            if (k < 0) break;                    // past the last output row
            const int i = select_in_frame(keep + (size_t)k * N, N, j - NA - before, lane);
            if (i < 0) break;                    // cannot happen when cnt matches keep
            f = k * N + i;
        }
        // (checked build: the output row and the source row both lie inside their F N rows)
        const bool row_ok = in_bounds(hdr, 4, j, (long long)F * N) && in_bounds(hdr, 4, f, (long long)F * N);
        if (lane < 3 && row_ok) {                // p_{k,i} = (k, y_i, x_i)  (Eq. compress_pos)
            const int k = f / N, i = f - k * N, yy = i / W;
            out_pos[(size_t)j * 3 + lane] = pos_base + (lane == 0 ? k + t_off : (lane == 1 ? yy : i - yy * W));
        }
        if (lane == 0 && !gave_up && row_ok) {
            for (int pc = 0; pc < pieces; ++pc) {
                const size_t off = (size_t)pc * kBulkPiece;
                const uint32_t bytes = (uint32_t)(row_bytes - off < (size_t)kBulkPiece ? row_bytes - off : kBulkPiece);
                bulk_wait_read<0>();             // the previous store has finished reading the buffer
                mbar_arrive_expect_tx(&bar[w], bytes + (uint32_t)tx_extra);
                if (stream_once) bulk_load_hint(buf, X + (size_t)f * row_bytes + off, bytes, &bar[w], once);
                else bulk_load(buf, X + (size_t)f * row_bytes + off, bytes, &bar[w]);
                if (!mbar_wait(&bar[w], phase & 1, wait_limit)) {
                    mbar_wait(&bar[w], phase & 1, wait_limit);   // one more bounded chance for the copy to land
                    gave_up = true;
                    break;
                }
                ++phase;
                if (stream_once == 2) bulk_store_hint(out_tokens + (size_t)j * row_bytes + off, buf, bytes, once);
                else bulk_store(out_tokens + (size_t)j * row_bytes + off, buf, bytes);
                bulk_commit();
            }
        }
        __syncwarp();
    }
    if (lane == 0) {
        bulk_wait<0>();                          // all rows of this warp are in global memory
        // L', or -1 if a wait of this call gave up.  Warp 0 has published L' above and looks at the error word now; a
        // warp that gave up raises the error word first and writes -1 afterwards.  Whichever order the two run in, -1
        // is what stays: either the -1 lands after L', or warp 0 sees the error word and writes -1 itself.
        if (gave_up) {
            report_give_up(hdr);
            __threadfence();
            *reinterpret_cast<volatile int*>(out_count) = -1;
        }
        if (gw == 0) {
            __threadfence();
            if (atomicAdd(hdr + HDR_ERROR, 0)) *reinterpret_cast<volatile int*>(out_count) = -1;
        }
    }
    trace_mark(hdr, 3, true);
}

// 32 keep flags (0 or 1 each) -> one bit each.  (The flags are masked first: a word that reaches past the end of the
// array holds other bytes, whose higher bits would spill into its neighbours' in the product.)
__device__ __forceinline__ unsigned pack_flags(const uint4& lo, const uint4& hi) {
    const unsigned w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    unsigned bits = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) bits |= ((((w[e] & 0x01010101u) * 0x01020408u) >> 24) & 0xfu) << (4 * e);   // byte i -> bit i
    return bits;
}
// position of the n-th (0-based) set bit; n < popcount(bits)
__device__ __forceinline__ int select_bit(unsigned bits, int n) {
    int at = 0;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const int c = __popc((bits >> at) & ((1u << h) - 1u));
        if (n >= c) { n -= c; at += h; }
    }
    return at;
}

// The same with the rows of a CTA found together.  A CTA owns a contiguous range of output rows.  It packs the keep
// flags of a window of tokens into bit words in shared memory together with the exclusive prefix of their population
// counts, after which the source row of any output row of the window is found by a binary search and a select in shared
// memory: the three dependent round trips (anchor, counts, flags) are paid once per window instead of once per row.
// Clips of up to kGatherWindow tokens need no survivor counts: the window is the whole clip.  Longer ones enter the walk
// at the frame that holds the CTA's first row and take as many windows, of a size that suits the range, as it needs.
//
// A warp moves a batch of consecutive output rows at a time, through two slots in turn, so that the next batch is on its
// way while this one lands: every lane issues the load of one row, and the batch leaves as one store, since the rows are
// contiguous in the output.  Rows longer than a slot go in pieces, a piece at a time.
//
// What bounds it where the GPU has nothing else to do is how soon the first copies are on their way: every CTA reads the same
// flags at the same moment, and they queue on the same cache lines of L2 (clock counts from the wait to the packed bits: 1100
// cycles with 29 CTAs on 1 KB of flags, 2150 with 141 on 3 KB, 2850 with 341 on 8 KB, 4250 with 444 on 13 KB; one row per
// warp at a time, which has every warp read counts and flags for itself, 5400 before its first copy).  Hence ONE CTA per SM
// there, and the slots as large as their sum may be: us per pass with three CTAs of 8 warps and 4 KB slots / one CTA of 16
// warps and 4 KB slots / one of 8 warps and 8 KB slots (128 KB both), in a replayed graph: 24 x 20 x 15 x 248 15.7 / 13.6 /
// 13.8, 32 x 16 x 16 x 2048 21.8 / 20.9 / 20.8, 64 x 32 x 32 x 1024 73.8 / 69.9 / 68.9, 128 x 32 x 32 x 64 27.7 / 27.7 / 28.6;
// from rows of 8 KB one at a time 9 x 16 x 16 x 4096 with a fixed anchor 20.9 / 20.2 / 15.4, 32 x 16 x 16 x 4096 32.8 / 31.4 /
// 30.9.  With 64 KB of slots 24 x 20 x 15 x 248 takes 16.8 and 32 x 16 x 16 x 4096 42.5, with 192 KB 13.7 and 32.7 (the
// sweep of the next call finds less L1).  Windows of 32768 or 65536 tokens gain nothing (128 x 16 x 16 x 512 22.1 / 22.3,
// 64 x 24 x 24 x 512 23.8 / 26.1).
// Where other clips' kernels run beside it the CTAs are three per SM, and long rows go one at a time: the waits of one CTA
// are filled by others (16 clips of 32 x 16 x 16 x 4096 448 us, 457 with one CTA per SM; 8 of 24 x 20 x 20 x 1024 84.6 / 87.4).
//
// WHOLE: the clip is one window.  Else the windows are `window_words` * 32 tokens.  NW: warps; `slot`: bytes of a staging slot, of
// which a warp has two; `pieces` of a row, or `batch` rows at most to a slot.
template <bool WHOLE, int NW>
__global__ void __launch_bounds__(NW * 32)
k_compact_rows(const __grid_constant__ ClipPtrs xs, size_t row_bytes, int F, int H, int W,
               int* __restrict__ hdr, const int* __restrict__ cnt, const int* __restrict__ gprefix,
               const unsigned char* __restrict__ keep, const __grid_constant__ OutPtrs outs, int NA, int acnt, int t_off,
               int pos_base, int late_trigger, int wait_limit, int tx_extra, int stream_once, size_t sstride, int window_words,
               unsigned per_magic, int pieces, int batch, int slot, int match_begins)
{
    constexpr int kThreads = NW * 32;
    const int words = WHOLE ? kGatherWords : window_words;
    const unsigned char* __restrict__ X = reinterpret_cast<const unsigned char*>(xs.X[blockIdx.y]);
    unsigned char* __restrict__ out_tokens = reinterpret_cast<unsigned char*>(outs.tokens[blockIdx.y]);
    int* __restrict__ out_pos = outs.pos[blockIdx.y];
    int* __restrict__ out_count = outs.count[blockIdx.y];
    hdr = clip_block(hdr, sstride); cnt = clip_block(cnt, sstride); gprefix = clip_block(gprefix, sstride);
    keep = clip_block(keep, sstride);

    extern __shared__ __align__(128) unsigned char stage[];     // [NW][2][slot]
    __shared__ uint64_t bar[NW][2];
    __shared__ unsigned s_bits[kGatherWords];
    __shared__ int s_pref[kGatherWords];
    __shared__ int s_warp[NW];
    __shared__ int s_frames[WHOLE ? 1 : kWarpPrefixMaxF + 4];
    const int N = H * W, FN = F * N;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (!late_trigger) pdl_launch_dependents();  // (see k_compact_bulk)
    trace_mark(hdr, 3, false);
    if (lane == 0) { mbar_init(&bar[w][0], 1); mbar_init(&bar[w][1], 1); mbar_init_fence(); }
    pdl_wait();                                  // keep flags and survivor counts are complete
    if (late_trigger) pdl_launch_dependents();
    trace_mark(hdr, 6, false);

    // ---- window of the walk: bits and prefix of tokens [T0, T0 + 32 words) ------------------------------------------
    constexpr int WPT = (kGatherWords + kThreads - 1) / kThreads;         // consecutive words per thread
    const int a = __ldcg(hdr + HDR_ANCHOR);
    const bool reporter = blockIdx.x == 0 && tid == 0;
    const int match_error = reporter && match_begins ? __ldcg(hdr + HDR_MATCH_ERROR) : 0;
    auto load_window = [&](int T0, int first) -> int {          // tokens before `first` do not count; returns the total
        uint4 v[WPT][2];
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
            const int f = T0 + (tid * WPT + u) * 32;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // (the flag array is 256-byte aligned and followed by other scratch: a load that starts inside it may
                // run past its end by less than 16 bytes, which the masks below discard)
                v[u][h] = tid * WPT < words && (unsigned)(f + h * 16) < (unsigned)FN ? __ldcg(reinterpret_cast<const uint4*>(keep + f) + h)
                                                                : make_uint4(0, 0, 0, 0);
            }
        }
        auto below = [](int n) -> unsigned { return n <= 0 ? 0u : (n >= 32 ? 0xffffffffu : (1u << n) - 1u); };
        unsigned b[WPT];
        int mine = 0;
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
            const int f = T0 + (tid * WPT + u) * 32;
            const unsigned anchor = below((a + 1) * N - f) & ~below(a * N - f);
            b[u] = pack_flags(v[u][0], v[u][1]);
            b[u] = acnt ? b[u] | anchor : b[u] & ~anchor;       // the anchor frame: all of its tokens, or none
            b[u] &= f < 0 || tid * WPT >= words ? 0u : below(FN - f) & ~below(first - f);          // (f < 0: past 2^31, hence past the end)
            mine += __popc(b[u]);
        }
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += n;
        }
        __syncthreads();                                        // (the window before this one is done with)
        if (lane == 31) s_warp[w] = incl;
        __syncthreads();
        int at = incl - mine, total = 0;
#pragma unroll
        for (int ww = 0; ww < NW; ++ww) { if (ww < w) at += s_warp[ww]; total += s_warp[ww]; }
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
            if (tid * WPT < words) {
                s_bits[tid * WPT + u] = b[u];
                s_pref[tid * WPT + u] = at;
            }
            at += __popc(b[u]);
        }
        __syncthreads();
        return total;
    };

    // ---- this CTA's rows [j0, j1) of the output ------------------------------------------------------------------
    const bool in_smem = F <= kWarpPrefixMaxF;   // (else the pre-scanned array)
    int k, before = 0, P, T0 = 0, in_window = 0;
    if (WHOLE) P = in_window = load_window(0, 0);      // (no survivor counts needed)
    else P = in_smem ? frame_prefix_cta<NW>(cnt, F, a, acnt, s_frames, s_warp) : __ldcg(gprefix + F);
    const int Lp = NA + P;                       // L' = N + P (Eq. Lpre)
    if (blockIdx.x == 0 && tid == 0) *reinterpret_cast<volatile int*>(out_count) = Lp;
    // rows per CTA: per_magic is 2^32 / gridDim.x rounded up, so that per * gridDim.x > Lp without a division (for one CTA
    // 2^32 - 1: per = Lp)
    const int per = (int)__umulhi((unsigned)Lp, per_magic) + 1;
    const int j0 = (int)min((long long)Lp, (long long)blockIdx.x * per), j1 = min(Lp, j0 + per);
    // rows per batch: what fits a slot, but no more than leaves every warp of the CTA a batch
    const int R = max(1, min(batch, (per + NW - 1) / NW));

    unsigned char* buf = stage + (size_t)w * 2 * slot;
    uint32_t phase = 0;                          // bit h: parity of slot h
    bool gave_up = false;                        // (lane 0 decides; all lanes of the warp know)
    const unsigned long long once = l2_evict_first_policy();

    auto source = [&](int j) {
        if (j < NA) return a * N + j;            // anchor rows first (Eq. xprime_stack)
        const int n = j - NA - before;           // the n-th token of the window: word by binary search, then the bit
        int lo = 0;
#pragma unroll
        for (int h = kGatherWords / 2; h > 0; h >>= 1) if ((WHOLE || h < words) && s_pref[lo + h] <= n) lo += h;
        return T0 + lo * 32 + select_bit(s_bits[lo], n - s_pref[lo]);
    };
    // A unit is a row, or a piece of a slot's size of a longer one.  Lanes 0 .. n-1 issue the loads of units ub .. ub + n - 1
    // behind output row jb into slot h and write the positions.
    auto unit_row = [&](int jb, int u, int& pc) {
        if (pieces == 1) { pc = 0; return jb + u; }
        const int r = u / pieces;
        pc = u - r * pieces;
        return jb + r;
    };
    auto unit_bytes = [&](int pc) { return (uint32_t)min(row_bytes - (size_t)pc * slot, (size_t)slot); };
    auto issue = [&](int jb, int ub, int n, int h) {
        if (lane == 0) {
            int pc;
            unit_row(jb, ub, pc);
            bulk_wait_read<0>();                 // the store that used this slot has finished reading it
            mbar_arrive_expect_tx(&bar[w][h], (uint32_t)n * unit_bytes(pc) + (uint32_t)tx_extra);
        }
        __syncwarp();
        if (lane < n) {
            int pc;
            const int j = unit_row(jb, ub + lane, pc), f = source(j);
            const bool ok = in_bounds(hdr, 4, j, FN) && in_bounds(hdr, 4, f, FN);      // (checked build)
            unsigned char* d = buf + h * slot + lane * (uint32_t)row_bytes;
            // (a row the checked build refuses is replaced by row 0, so that the batch still completes)
            const unsigned char* src = X + (size_t)(ok ? f : 0) * row_bytes + (size_t)pc * slot;
            if (stream_once) bulk_load_hint(d, src, unit_bytes(pc), &bar[w][h], once);
            else bulk_load(d, src, unit_bytes(pc), &bar[w][h]);
            if (ok && pc == 0) {                 // p_{k,i} = (k, y_i, x_i)  (Eq. compress_pos)
                const int kk = f / N, i = f - kk * N, yy = i / W;
                int* p = out_pos + (size_t)j * 3;
                p[0] = pos_base + kk + t_off; p[1] = pos_base + yy; p[2] = pos_base + i - yy * W;
            }
        }
    };
    auto finish = [&](int jb, int ub, int n, int h) {            // the batch has landed: one store
        if (lane == 0) {
            int pc;
            const int j = unit_row(jb, ub, pc);
            if (!mbar_wait(&bar[w][h], (phase >> h) & 1, wait_limit)) {
                mbar_wait(&bar[w][h], (phase >> h) & 1, wait_limit);     // one more bounded chance for the copies to land
                gave_up = true;
            } else if (in_bounds(hdr, 4, j + (pieces == 1 ? n - 1 : 0), FN)) {
                unsigned char* d = out_tokens + (size_t)j * row_bytes + (size_t)pc * slot;
                if (stream_once == 2) bulk_store_hint(d, buf + h * slot, (uint32_t)n * unit_bytes(pc), once);
                else bulk_store(d, buf + h * slot, (uint32_t)n * unit_bytes(pc));
                bulk_commit();
            }
        }
        phase ^= 1u << h;
        gave_up = __shfl_sync(0xffffffffu, gave_up ? 1 : 0, 0) != 0;
    };
    auto move_rows = [&](int ja, int jb) {       // rows [ja, jb) of the output, by the warps of the CTA in turn
        const int units = (jb - ja) * pieces;
        int at = w * R, h = 0;
        if (at < units && !gave_up) issue(ja, at, min(R, units - at), 0);
        for (; at < units && !gave_up; at += NW * R) {
            const int next = at + NW * R;
            if (next < units) issue(ja, next, min(R, units - next), h ^ 1);
            finish(ja, at, min(R, units - at), h);
            h ^= 1;
        }
    };

    if (WHOLE) move_rows(j0, j1);
    else {
        move_rows(j0, min(j1, NA));
        int e = max(j0, NA) - NA;                // next token of the walk this CTA emits
        const int e1 = j1 - NA;
        if (e < e1) {                            // (e, e1 and the counts are the same for all threads)
            if (in_smem) { k = frame_of(s_frames, F, e); before = s_frames[k]; }
            else find_frame(cnt, gprefix, F, a, acnt, lane, e, k, before);
            T0 = (k * N) & ~31;
            in_window = load_window(T0, k * N);
        }
        while (e < e1) {
            const int upto = min(e1, before + in_window);
            move_rows(NA + e, NA + upto);
            e = upto;
            if (e >= e1 || T0 >= FN - words * 32) break;      // (the second cannot happen when the counts match the flags)
            before += in_window;
            T0 += words * 32;
            in_window = load_window(T0, 0);
        }
    }

    if (lane == 0) {
        if (gave_up)                             // copies still on their way into this CTA's shared memory (bounded again)
            for (int h = 0; h < 2; ++h) mbar_wait(&bar[w][h], (phase >> h) & 1, wait_limit);
        bulk_wait<0>();                          // all rows of this warp are in global memory
        if (gave_up) {                           // L' or -1: see k_compact_bulk
            report_give_up(hdr);
            __threadfence();
            *reinterpret_cast<volatile int*>(out_count) = -1;
        }
        if (reporter) {
            if (match_error) {                   // (a matching kernel that began its call)
                report_give_up(hdr);
                hdr[HDR_MATCH_ERROR] = 0;
            }
            __threadfence();
            if (atomicAdd(hdr + HDR_ERROR, 0)) *reinterpret_cast<volatile int*>(out_count) = -1;
        }
    }
    trace_mark(hdr, 3, true);
}

template <int COPY_BYTES>
__global__ void __launch_bounds__(kCopyWarps * 32)
k_compact(const __grid_constant__ ClipPtrs xs, size_t row_bytes, int F, int H, int W,
          const int* __restrict__ hdr, const int* __restrict__ cnt, const int* __restrict__ gprefix,
          const unsigned char* __restrict__ keep, const __grid_constant__ OutPtrs outs, int NA, int acnt, int t_off,
          int pos_base, int late_trigger, size_t sstride)
{
    const unsigned char* __restrict__ X = reinterpret_cast<const unsigned char*>(xs.X[blockIdx.y]);
    unsigned char* __restrict__ out_tokens = reinterpret_cast<unsigned char*>(outs.tokens[blockIdx.y]);
    int* __restrict__ out_pos = outs.pos[blockIdx.y];
    int* __restrict__ out_count = outs.count[blockIdx.y];
    hdr = clip_block(hdr, sstride); cnt = clip_block(cnt, sstride); gprefix = clip_block(gprefix, sstride);
    keep = clip_block(keep, sstride);
    using U = typename CopyUnit<COPY_BYTES>::type;
    const int N = H * W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    trace_mark(const_cast<int*>(hdr), 3, false);
    if (!late_trigger) pdl_launch_dependents();  // (see k_compact_bulk)
    pdl_wait();                                  // keep flags, dst and survivor counts are complete
    if (late_trigger) pdl_launch_dependents();
    trace_mark(const_cast<int*>(hdr), 6, false);
    const int a = __ldcg(hdr + HDR_ANCHOR);

    // ---- output-driven gather, one warp per output row, no block-level synchronisation -----------------------
    // frame search: the frame that holds the e-th preserved source token (flat order, anchor frame skipped)
    // and the number of preserved tokens before that frame.  Returns the total P when e is past the end.
    const int gw = blockIdx.x * kCopyWarps + w;            // global warp index
    const int nw = gridDim.x * kCopyWarps;
    if (gw == 0) {                                         // L' = N + P (Eq. Lpre)
        int kk, bb;
        const int P = find_frame(cnt, gprefix, F, a, acnt, lane, -1, kk, bb);
        // a bounded wait of an earlier kernel of this call gave up: report instead of a plausible count
        if (lane == 0) *out_count = __ldcg(hdr + HDR_ERROR) ? -1 : NA + P;
    }
    const int upr = (int)(row_bytes / COPY_BYTES);         // copy units per row
    for (int j = gw; ; j += nw) {
        int f;
        if (j < NA) f = a * N + j;                         // anchor rows first (Eq. xprime_stack)
        else {
            int k, before;
            find_frame(cnt, gprefix, F, a, acnt, lane, j - NA, k, before);
            if (k < 0) break;                              // past the last output row
            const int i = select_in_frame(keep + (size_t)k * N, N, j - NA - before, lane);
            if (i < 0) break;                              // cannot happen when cnt matches keep
            f = k * N + i;
        }
        const bool row_ok = in_bounds(const_cast<int*>(hdr), 4, j, (long long)F * N) &&
                            in_bounds(const_cast<int*>(hdr), 4, f, (long long)F * N);     // (checked build)
        if (!row_ok) continue;
        if (lane < 3) {                                    // p_{k,i} = (k, y_i, x_i)  (Eq. compress_pos)
            const int k = f / N, i = f - k * N, yy = i / W;
            out_pos[(size_t)j * 3 + lane] = pos_base + (lane == 0 ? k + t_off : (lane == 1 ? yy : i - yy * W));
        }
        const U* src = reinterpret_cast<const U*>(X + (size_t)f * row_bytes);
        U* dsto = reinterpret_cast<U*>(out_tokens + (size_t)j * row_bytes);
        for (int u0 = lane; u0 < upr; u0 += 32 * kCopyUnroll) {
            U v[kCopyUnroll];
#pragma unroll
            for (int q = 0; q < kCopyUnroll; ++q) if (u0 + q * 32 < upr) v[q] = __ldcs(src + u0 + q * 32);
#pragma unroll
            for (int q = 0; q < kCopyUnroll; ++q) if (u0 + q * 32 < upr) __stcs(dsto + u0 + q * 32, v[q]);
        }
    }
    trace_mark(const_cast<int*>(hdr), 3, true);
}

cudaError_t launch_compact(const Problem& p, const Scratch& s, const OutPtrs& out, cudaStream_t st) {
    const size_t esize = p.dtype == 0 ? 4 : 2;
    const size_t row_bytes = (size_t)p.C * esize;
    bool vec = p.vec;
    for (int n = 0; n < p.nclips; ++n) vec = vec && reinterpret_cast<uintptr_t>(out.tokens[n]) % 16 == 0;
    // rows emitted as the anchor block / tokens the anchor frame adds to the flat walk: (N, 0) in the paper's order
    // (Eq. xprime_stack), (0, N) in natural order, (0, 0) for a streaming segment, which does not emit its anchor
    const int NA = (p.emit_anchor && !p.natural_order) ? p.N : 0;
    const int acnt = (p.emit_anchor && p.natural_order) ? p.N : 0;
    if (p.F > kWarpPrefixMaxF) {
        k_frame_prefix<<<dim3(1, p.nclips), 1024, 0, st>>>(s.cnt, s.hdr, p.F, acnt, s.prefix, p.sstride);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // enough warps for one output row each at the usual two-thirds removal, at most three CTAs per SM and clip (a warp
    // loops when there are more)
    const long long want = ((long long)p.F * p.N / 3 + p.N + kCopyWarps - 1) / kCopyWarps;
    const int grid = (int)(want < 3LL * sm_count() ? (want < 1 ? 1 : want) : 3LL * sm_count());
    const dim3 b(kCopyWarps * 32);
    // the pre-scanned prefix of very long clips is read through plain loads: order that case by the stream
    const bool pdl = p.F <= kWarpPrefixMaxF;
    // Beside other clips' kernels, short rows in batches: up to half a slot always, up to a slot where the clip is one window of
    // flags.  Measured, us per pass with one row per warp at a time / with batches: 128 x 32 x 32 x 64 (128-byte rows) 89.3 / 44.1,
    // 128 x 24 x 24 x 256 58.5 / 39.6, 64 x 24 x 24 x 512 43.7 / 35.6, 64 x 32 x 32 x 1024 93.2 / 80.9; 4096-byte rows:
    // 32 x 16 x 16 (one window) 29.3 / 28.5, 128 x 16 x 16 (two windows) 74.6 / 78.4; 2320-byte rows, one window
    // 23.2 / 21.7.  Longer rows keep every warp's slot full by themselves.
    const long long FN = (long long)p.F * p.N;
    const bool whole = FN <= kGatherWindow;
    const bool alone = gather_alone(p);
    if (vec && (alone || row_bytes <= 2048 || (row_bytes <= 4096 && whole))) {
        auto launch = [&](auto kernel, int nw, int slot, int per_sm) {
            const size_t smem = (size_t)nw * 2 * slot;
            const int ctas = (int)std::min((FN / 3 + p.N + nw - 1) / nw, std::max(1LL, (long long)per_sm * sm_count() / p.nclips));
            const int pieces = (int)((row_bytes + slot - 1) / slot);
            const int batch = pieces > 1 ? 1 : (int)std::min((size_t)32, slot / row_bytes);
            const unsigned per_magic = ctas == 1 ? 0xffffffffu : (unsigned)(((1ULL << 32) + ctas - 1) / ctas);
            // Clips beyond one window: windows of sixteen times the tokens that fall to a CTA (a window that holds too few rows
            // costs another round trip), at least 512.  (Against windows of 16384 tokens and a count prefix per warp, us per
            // pass: 64 x 24 x 24 x 512 32.3 -> 30.6, 64 x 32 x 32 x 1024 76.8 -> 75.2, 128 x 32 x 32 x 64 31.8 -> 29.8.  Clips
            // of one window are better off without the counts: 32 x 16 x 16 x 2048 27.0 against 28.0.)
            int words = 16;
            while (words < kGatherWords && words * 32LL < 16 * FN / ctas) words *= 2;
            cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
            if (e != cudaSuccess) return e;
            return launch_ex(pdl, smem, kernel, dim3(ctas, p.nclips), dim3(nw * 32), st, p.xs, row_bytes, p.F, p.H, p.W, s.hdr,
                             (const int*)s.cnt, (const int*)s.prefix, (const unsigned char*)s.keep, out, NA, acnt,
                             p.pos_t_offset, p.pos_base, p.chain_next, wait_poll_limit(), wait_tx_extra(), p.stream_once,
                             p.sstride, words, per_magic, pieces, batch, slot, p.match_begins);
        };
        if (!alone) return whole ? launch(k_compact_rows<true, 8>, 8, 4096, 3) : launch(k_compact_rows<false, 8>, 8, 4096, 3);
        if (row_bytes <= 128)                    // (32 rows, one per lane, fill no more than half a slot of 8 KB)
            return whole ? launch(k_compact_rows<true, 16>, 16, 4096, 1) : launch(k_compact_rows<false, 16>, 16, 4096, 1);
        return whole ? launch(k_compact_rows<true, 8>, 8, 8192, 1) : launch(k_compact_rows<false, 8>, 8, 8192, 1);
    }
    const dim3 g(grid, p.nclips);
    if (vec) {
        const size_t smem = (size_t)kCopyWarps * kBulkPiece;
        cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_compact_bulk), smem);
        if (e != cudaSuccess) return e;
        return launch_ex(pdl, smem, k_compact_bulk, g, b, st, p.xs, row_bytes, p.F, p.H, p.W, s.hdr, (const int*)s.cnt,
                         (const int*)s.prefix, (const unsigned char*)s.keep, out, NA, acnt, p.pos_t_offset, p.pos_base,
                         p.chain_next, wait_poll_limit(), wait_tx_extra(), p.stream_once, p.sstride);
    }
    if (esize == 4)
        return launch_pdl_if(pdl, k_compact<4>, g, b, st, p.xs, row_bytes, p.F, p.H, p.W, (const int*)s.hdr,
                             (const int*)s.cnt, (const int*)s.prefix, (const unsigned char*)s.keep, out, NA, acnt,
                             p.pos_t_offset, p.pos_base, p.chain_next, p.sstride);
    return launch_pdl_if(pdl, k_compact<2>, g, b, st, p.xs, row_bytes, p.F, p.H, p.W, (const int*)s.hdr,
                         (const int*)s.cnt, (const int*)s.prefix, (const unsigned char*)s.keep, out, NA, acnt,
                         p.pos_t_offset, p.pos_base, p.chain_next, p.sstride);
}

}  // namespace ttf
