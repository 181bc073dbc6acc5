// Step (c) (Sec. 3.2): the u positions with the largest M~ among i < L, equal values ordered by
// position, written in ascending position order.  A block-wide routine shared by the stand-alone
// select kernel and the fused forward kernel.
#pragma once
#include "psattn_common.cuh"

namespace psattn {

constexpr int kSelectMaxSlots = 18;       // keys per thread of block_select_few at most
constexpr int kSelectCands = 240;         // its candidates at most

struct SelectScratch {
    int hist[256];
    int wtot_gt[32], wtot_eq[32];
    int wpre_gt[33], wpre_eq[33];
    unsigned prefix;
    int remaining;
    int done;
    // block_select_short
    uint2 count[2][32];                                    // warp totals of a round (two rounds in turn)
    unsigned lo[32], hi[32];
    unsigned taken[8][32];                                 // per key slot and warp: keys above tau, keys equal to it << 16
    // block_select_few
    uint2 cand[kSelectCands];                              // key, position
    unsigned char in[kSelectCands];
    int n_cand;
};

// The first nthr threads of the block (whole warps, which meet at the named barrier; 0 and blockDim.x: all) call this with
// the same arguments.
// key_of(i) returns the order-preserving key of position i (larger key = larger M~); it is called
// several times per position and must be cheap (a global or shared-memory read).
// Four 8-bit radix passes find tau, the u-th largest key; the result is every position with
// key > tau plus the first `remaining` positions with key == tau.  out[0..u_max) receives the
// positions in ascending order, -1 padded.  Ends with a __syncthreads().
template <class KeyFn>
__device__ __forceinline__ void block_select(KeyFn key_of, int L, int u, int u_max, int *out, SelectScratch &s, int nthr, int barrier) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nthr >> 5;
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(nthr) : "memory"); };
    if (u <= 0) {
        for (int r = tid; r < u_max; r += nthr) out[r] = -1;
        sync();
        return;
    }
    if (tid == 0) { s.prefix = 0u; s.remaining = u; s.done = 0; }
    unsigned known = 0u;                                   // key bits fixed so far
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int t = tid; t < 256; t += nthr) s.hist[t] = 0;
        sync();
        const unsigned prefix = s.prefix;
        for (int i = tid; i < L; i += nthr) {
            const unsigned k = key_of(i);
            if (((k ^ prefix) & known) == 0u) atomicAdd(&s.hist[(k >> shift) & 255u], 1);
        }
        sync();
        if (wid == 0) {                                    // find the bin that holds the remaining-th largest
            int h[8], mine = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { h[j] = s.hist[lane * 8 + j]; mine += h[j]; }
            int incl = mine;                               // becomes the count of bins >= this lane's first bin
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_down_sync(0xffffffffu, incl, o);
                if (lane + o < 32) incl += y;
            }
            const int above = incl - mine, rem = s.remaining;
            __syncwarp();
            if (above < rem && incl >= rem) {              // exactly one lane
                int r = rem - above, bin = 7;
                for (; bin > 0; --bin) {
                    if (h[bin] >= r) break;
                    r -= h[bin];
                }
                const unsigned value = prefix | ((unsigned)(lane * 8 + bin) << shift);
                if (h[bin] == r && value != 0u) {
                    // every key of this bin is taken: the result is "all keys >= value"; no need to
                    // resolve the lower bits
                    s.prefix = value - 1u;
                    s.remaining = 0;
                    s.done = 1;
                } else {
                    s.prefix = value;
                    s.remaining = r;
                }
            }
        }
        known |= 0xffu << shift;
        sync();
        if (s.done) break;
    }
    const unsigned tau = s.prefix;
    const int need_eq = s.remaining;                       // positions with key == tau to take, lowest first
    int gt_seen = 0, eq_seen = 0;
    for (int base = 0; base < L; base += nthr) {
        const int i = base + tid;
        const bool valid = i < L;
        const unsigned k = valid ? key_of(i) : 0u;
        const int is_gt = valid && k > tau, is_eq = valid && k == tau;
        int xg = is_gt, xe = is_eq;                        // inclusive warp scans of both flags
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int yg = __shfl_up_sync(0xffffffffu, xg, o), ye = __shfl_up_sync(0xffffffffu, xe, o);
            if (lane >= o) { xg += yg; xe += ye; }
        }
        if (lane == 31) { s.wtot_gt[wid] = xg; s.wtot_eq[wid] = xe; }
        sync();
        if (wid == 0) {                                        // exclusive scan of the warp totals; grand totals in [nw]
            int tg = lane < nw ? s.wtot_gt[lane] : 0, te = lane < nw ? s.wtot_eq[lane] : 0;
            const int og = tg, oe = te;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int yg = __shfl_up_sync(0xffffffffu, tg, o), ye = __shfl_up_sync(0xffffffffu, te, o);
                if (lane >= o) { tg += yg; te += ye; }
            }
            s.wpre_gt[lane] = tg - og; s.wpre_eq[lane] = te - oe;
            if (lane == 31) { s.wpre_gt[32] = tg; s.wpre_eq[32] = te; }
        }
        sync();
        const int bg = s.wpre_gt[wid], be = s.wpre_eq[wid], tg = s.wpre_gt[32], te = s.wpre_eq[32];
        const int gt_before = gt_seen + bg + xg - is_gt, eq_before = eq_seen + be + xe - is_eq;
        // taken positions before this one: all greater ones, and the equal ones up to need_eq
        if (is_gt || (is_eq && eq_before < need_eq)) {
            const int pos = gt_before + min(eq_before, need_eq);
            if (pos < u_max) out[pos] = i;
        }
        gt_seen += tg; eq_seen += te;
        sync();
    }
    for (int r = u + tid; r < u_max; r += nthr) out[r] = -1;
    sync();
}

// The same selection for lists that fit the block's registers (L <= KPT * nthr): every thread keeps its keys
// (positions tid, tid + nthr, ...) and the block bisects the key range for tau.  A round counts the keys at or above three
// thresholds across the block; it ends as soon as exactly u keys lie at or above one, which takes as many rounds as the
// key range is wider, in powers of four, than the gap below the u-th largest: five or six for 1024 values, against three
// radix passes whose shared-memory atomics pile up in the few bins that keys of like exponent share.  Selection phase of
// the fused kernel, with the ordered write-out: 2.7 -> 1.9 us at T = 64 .. 203, 3.8 -> 2.6 us at T = 1024.
// Called by the first nthr threads of the block (whole warps), which meet at the named barrier (0, blockDim.x: all).
template <int KPT, class KeyFn>
__device__ __forceinline__ void block_select_short(KeyFn key_of, int L, int u, int u_max, int *out, SelectScratch &s, int nthr,
                                                   int barrier) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nthr >> 5;
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(nthr) : "memory"); };
    if (u <= 0) {
        for (int r = tid; r < u_max; r += nthr) out[r] = -1;
        sync();
        return;
    }
    unsigned key[KPT];
    unsigned mn = 0xffffffffu, mx = 0u;
#pragma unroll
    for (int x = 0; x < KPT; ++x) {
        const int i = tid + x * nthr;
        key[x] = 0u;
        if (i < L) { key[x] = key_of(i); mn = min(mn, key[x]); mx = max(mx, key[x]); }
    }
    mn = __reduce_min_sync(0xffffffffu, mn); mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) { s.lo[wid] = mn; s.hi[wid] = mx; }
    sync();
    // tau = the largest threshold with at least u keys at or above it: lo always has them, hi + 1 has `above` < u
    unsigned lo = __reduce_min_sync(0xffffffffu, lane < nw ? s.lo[lane] : 0xffffffffu);
    unsigned hi = __reduce_max_sync(0xffffffffu, lane < nw ? s.hi[lane] : 0u);
    int above = 0;
    bool exact = L == u;                                   // exactly u keys >= lo
    for (int round = 0; lo < hi && !exact; round ^= 1) {   // three thresholds a round: a quarter of the range is left
        const unsigned w = hi - lo, step = (w >> 2) + 1u;
        const unsigned t1 = lo + step, t2 = lo + min(2u * step, w), t3 = lo + min(3u * step, w);
        unsigned c12 = 0u, c3 = 0u;
#pragma unroll
        for (int x = 0; x < KPT; ++x)
            if (tid + x * nthr < L) {
                c12 += (key[x] >= t1 ? 1u : 0u) + (key[x] >= t2 ? 0x10000u : 0u);
                c3 += key[x] >= t3 ? 1u : 0u;
            }
        c12 = __reduce_add_sync(0xffffffffu, c12); c3 = __reduce_add_sync(0xffffffffu, c3);
        if (lane == 0) s.count[round][wid] = make_uint2(c12, c3);
        sync();
        const uint2 v = lane < nw ? s.count[round][lane] : make_uint2(0u, 0u);
        c12 = __reduce_add_sync(0xffffffffu, v.x);
        const int n3 = (int)__reduce_add_sync(0xffffffffu, v.y), n2 = (int)(c12 >> 16), n1 = (int)(c12 & 0xffffu);
        if (n3 >= u) { lo = t3; exact = n3 == u; }
        else if (n2 >= u) { lo = t2; hi = t3 - 1u; above = n3; exact = n2 == u; }
        else if (n1 >= u) { lo = t1; hi = t2 - 1u; above = n2; exact = n1 == u; }
        else { hi = t1 - 1u; above = n1; }
    }
    // Taken: the keys > lo, and of those == lo the first need_eq by position (all of them when exactly u are >= lo).
    // Position order is (x, warp, lane): totals per x and warp give every position its place.
    const int need_eq = exact ? L : u - above;
#pragma unroll
    for (int x = 0; x < KPT; ++x) {
        if (x * nthr >= L) break;
        const bool valid = tid + x * nthr < L;
        const unsigned bg = __ballot_sync(0xffffffffu, valid && key[x] > lo), be = __ballot_sync(0xffffffffu, valid && key[x] == lo);
        if (lane == 0) s.taken[x][wid] = (unsigned)__popc(bg) | (unsigned)__popc(be) << 16;
    }
    sync();
    unsigned seen = 0u;
#pragma unroll
    for (int x = 0; x < KPT; ++x) {
        if (x * nthr >= L) break;
        const int i = tid + x * nthr;
        const bool gt = i < L && key[x] > lo, eq = i < L && key[x] == lo;
        const unsigned lower = (1u << lane) - 1u;
        const unsigned mine = (unsigned)__popc(__ballot_sync(0xffffffffu, gt) & lower) |
                              (unsigned)__popc(__ballot_sync(0xffffffffu, eq) & lower) << 16;
        const unsigned tot = lane < nw ? s.taken[x][lane] : 0u;
        const unsigned before = seen + mine + __reduce_add_sync(0xffffffffu, lane < wid ? tot : 0u);
        const int g0 = (int)(before & 0xffffu), e0 = (int)(before >> 16);
        if (gt || (eq && e0 < need_eq)) {
            const int pos = g0 + min(e0, need_eq);
            if (pos < u_max) out[pos] = i;
        }
        seen += __reduce_add_sync(0xffffffffu, tot);
    }
    for (int r = u + tid; r < u_max; r += nthr) out[r] = -1;
    sync();
}

// The selection for small u (u <= 64 < nthr) in two steps: the u-th largest of the threads' own maxima bounds tau from below,
// so the few keys at or above it hold the top u; these are ranked against each other by (key, position), which settles ties
// too.  The bound may be loose (up to kSlack keys too many), which saves rounds of the search.  Many equal keys can overflow the
// candidates; then key_of is asked again and block_select takes over.  Called by the first nthr threads (whole warps).
// For the long lists (18 keys per thread): selection phase at T = 8192 9.9 -> 6.5 us, T = 4000 6.3 -> 4.4 us against
// block_select_short, which is the faster one up to about 1000 keys (2.2 against 2.3 us at T = 512).
template <int KPT, class KeyFn>
__device__ __forceinline__ void block_select_few(KeyFn key_of, int L, int u, int u_max, int *out, SelectScratch &s, int nthr,
                                                 int barrier) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nthr >> 5;
    constexpr int kSlack = 32;
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(nthr) : "memory"); };
    for (int r = u + tid; r < u_max; r += nthr) out[r] = -1;
    if (u <= 0) { sync(); return; }
    unsigned key[KPT], top = 0u;
#pragma unroll
    for (int x = 0; x < KPT; ++x) {
        const int i = tid + x * nthr;
        key[x] = i < L ? key_of(i) : 0u;
        top = max(top, key[x]);
    }
    const bool owns = tid < L;                             // this thread has keys
    unsigned lo = 0u, hi = 0u;
    {
        const unsigned mn = __reduce_min_sync(0xffffffffu, owns ? top : 0xffffffffu), mx = __reduce_max_sync(0xffffffffu, top);
        if (lane == 0) { s.lo[wid] = mn; s.hi[wid] = mx; }
        if (tid == 0) s.n_cand = 0;
        sync();
        lo = __reduce_min_sync(0xffffffffu, lane < nw ? s.lo[lane] : 0xffffffffu);
        hi = __reduce_max_sync(0xffffffffu, lane < nw ? s.hi[lane] : 0u);
    }
    // invariant: at least u maxima are >= lo, fewer than u are > hi
    bool near = min(L, nthr) <= u + kSlack;
    for (int round = 0; lo < hi && !near; round ^= 1) {
        const unsigned w = hi - lo, step = (w >> 2) + 1u;
        const unsigned t1 = lo + step, t2 = lo + min(2u * step, w), t3 = lo + min(3u * step, w);
        const unsigned b1 = __ballot_sync(0xffffffffu, owns && top >= t1), b2 = __ballot_sync(0xffffffffu, owns && top >= t2),
                       b3 = __ballot_sync(0xffffffffu, owns && top >= t3);
        if (lane == 0) s.count[round][wid] = make_uint2((unsigned)__popc(b1) | (unsigned)__popc(b2) << 16, (unsigned)__popc(b3));
        sync();
        const uint2 v = lane < nw ? s.count[round][lane] : make_uint2(0u, 0u);
        const unsigned c12 = __reduce_add_sync(0xffffffffu, v.x);
        const int n3 = (int)__reduce_add_sync(0xffffffffu, v.y), n2 = (int)(c12 >> 16), n1 = (int)(c12 & 0xffffu);
        if (n3 >= u) { lo = t3; near = n3 <= u + kSlack; }
        else if (n2 >= u) { lo = t2; hi = t3 - 1u; near = n2 <= u + kSlack; }
        else if (n1 >= u) { lo = t1; hi = t2 - 1u; near = n1 <= u + kSlack; }
        else hi = t1 - 1u;
    }
    if (owns && top >= lo) {
#pragma unroll
        for (int x = 0; x < KPT; ++x)
            if (tid + x * nthr < L && key[x] >= lo) {
                const int at = atomicAdd(&s.n_cand, 1);
                if (at < kSelectCands) s.cand[at] = make_uint2(key[x], (unsigned)(tid + x * nthr));
            }
    }
    sync();
    const int n = s.n_cand;
    if (n > kSelectCands) {                                // (uniform)
        block_select(key_of, L, u, u_max, out, s, nthr, barrier);
        return;
    }
    // four lanes per candidate: how many come before it by (key descending, position); then, of those taken, by position
    const int part = tid & 3;
    for (int c0 = 0; c0 < n; c0 += nthr >> 2) {
        const int c = c0 + (tid >> 2);
        const uint2 me = c < n ? s.cand[c] : make_uint2(0u, 0u);
        int before = 0;
#pragma unroll 4
        for (int o = part; o < n; o += 4) {
            const uint2 x = s.cand[o];
            before += x.x > me.x || (x.x == me.x && x.y < me.y);
        }
        before += __shfl_xor_sync(0xffffffffu, before, 1);
        before += __shfl_xor_sync(0xffffffffu, before, 2);
        if (part == 0 && c < n) s.in[c] = before < u;
    }
    sync();
    for (int c0 = 0; c0 < n; c0 += nthr >> 2) {
        const int c = c0 + (tid >> 2);
        const unsigned pos = c < n ? s.cand[c].y : 0u;
        int before = 0;
#pragma unroll 4
        for (int o = part; o < n; o += 4) before += s.in[o] && s.cand[o].y < pos;
        before += __shfl_xor_sync(0xffffffffu, before, 1);
        before += __shfl_xor_sync(0xffffffffu, before, 2);
        if (part == 0 && c < n && s.in[c] && before < u_max) out[before] = (int)pos;
    }
    sync();
}

}  // namespace psattn
