// The whole path (steps a-e) of one (batch, head) unit in one launch for fp32 inputs: psattn_fused.cu's plan in fp32
// arithmetic on the FMA pipe (tf32 products would break the 1e-4 tolerance).
//
//   1. the unit's keys into shared memory where they fit (T up to about 870), then the measure, one warp per query (Eq. 11)
//   2. block-wide selection                                                                        (Sec. 3.2)
//   3. attention of the selected rows: chunks of 128 keys, scores in 8 x 2 register tiles, softmax, values in 4 x 4 register
//      tiles with the keys of the chunk spread over the threads that the rows leave free; a zero query row
//      yields the column sums of V                                                                 (Eq. 7-8)
//   4. fill                                                                                        (Eq. 12)
// A unit is shared by the CTAs of a cluster as in psattn_fused.cu.
// Bound: the measure's row reads (256 bytes per pair from shared memory at 128 B/clk), then latency.  The staged schedule ran
// five kernels, of which the attention gave every (row, key split) to one warp that read all keys and values for itself: 99 us
// of the 136 us at B8 H4 T777 (lengths 233..777), 14 of 29 us for B1 H4 T128.
#include "psattn_cluster.cuh"
#include "psattn_launch.h"
#include "psattn_measure_mma.cuh"
#include "psattn_select.cuh"

namespace psattn {

using namespace sm100;

constexpr int kF32Threads = 512;
constexpr int kF32MaxRows = 64;
constexpr int kF32Chunk = 128;                                 // keys per step of the attention
constexpr int kF32KPitch = 68, kF32PPitch = 72;                // floats: conflict-free 16-byte reads of eight rows; 16-byte rows
constexpr uint32_t kF32OffQ = 0;                               // [64][64]
constexpr uint32_t kF32OffK = kF32OffQ + 64 * 64 * 4;          // [128][68]
constexpr uint32_t kF32OffV = kF32OffK + kF32Chunk * kF32KPitch * 4;       // [128][64]; afterwards the row states
constexpr uint32_t kF32OffP = kF32OffV + kF32Chunk * 64 * 4;   // [128][72]: weights, key-major; afterwards partial sums
constexpr uint32_t kF32AttendBytes = kF32OffP + kF32Chunk * kF32PPitch * 4;
constexpr size_t kF32MaxSmem = 226 * 1024;

struct Fused32Args {
    uint32_t off_persist;                // M~, selection, flags: live through all phases
    int resident;                        // the unit's keys fit in shared memory
    int own_v, by_length, split, m_floats;
    const int *sel_in;
};

struct Fused32Persist {
    SelectScratch select;
    int sel[kF32MaxRows];
    float vbar[kD];
    float m[2][kF32MaxRows], l[kF32MaxRows];       // references before and after a chunk, in turn
    float part[kF32MaxRows][2], sum[kF32MaxRows][2];         // row maxima and row sums of the two warps of a row group
    int b_ranked;
};

__host__ __device__ inline size_t f32_arrays_bytes(int m_floats, int T) { return ((size_t)4 * m_floats + T + 127) / 128 * 128; }

// acc += (a0 b0, a1 b1) in one instruction
__device__ __forceinline__ void f32_fma2(float2 &acc, float a0, float a1, float b0, float b1) {
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%0, %1};\n\t"
        "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "+f"(acc.x), "+f"(acc.y) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// One query's samples, kept one query ahead: its row (8 columns per lane) and up to 64 key positions.
struct F32Query {
    float q[8];
    int key[2];
};

// M~ of the queries q_lo + warp, + 16, ... < q_hi of one unit.  Four groups of eight lanes, a group takes every fourth sampled
// key (lane `sub` its columns 8 sub .. 8 sub + 7); 16 keys are in flight, and their 16 dot products are summed over the
// eight lanes by exchanging halves (four shuffles instead of twelve), after which lane (grp, sub) holds the score of
// sample 16 n + 4 x + grp, x = 2 (sub & 1) + (sub >> 1 & 1).  At most 64 samples, so all scores of a query stay in
// registers: M~ = (1/U) sum_j (max - s_j) exactly as written, never negative and 0 for equal scores.
// Resident rows hold their 16-byte piece c at c ^ (c >> 3): the even pieces of a row lie in eight different bank groups, and
// so do the odd ones.
// NB = ceil(U / 16) batches, straight-line, so that the loads of one run under the sums of another.
template <bool RESIDENT, int NB>
__device__ __forceinline__ void f32_measure_n(const Geom &g, int unit, int b, int h, int L, int U, int q_lo, int q_hi,
                                            const float *__restrict__ Qu, const float *Ku, long long k_pitch,
                                            const int *__restrict__ sidx, float *M_s) {
    const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3, warp = threadIdx.x >> 5;
    const int *idx0 = sidx + (g.idx_per_head ? (long long)unit : (long long)b) * g.T * g.idx_cols;
    const float4 *Kl = reinterpret_cast<const float4 *>(Ku) + (RESIDENT ? 0 : 2 * sub);    // (dense shared rows: 32-bit indices)
    const int at_lo = 2 * sub ^ (sub >> 2), at_hi = (2 * sub + 1) ^ (sub >> 2);
    const int mine = 4 * (2 * (sub & 1) + ((sub >> 1) & 1)) + grp;         // this lane's sample in a batch of 16
    const bool b0 = sub & 1, b1 = sub & 2;
    auto fetch = [&](int i, F32Query &x) {
        if (i >= q_hi) return;
        load8(Qu + (long long)i * g.qs[2], sub, x.q);
        const int *row = idx0 + (long long)i * g.idx_cols;
        x.key[0] = lane < U ? __ldg(row + lane) : 0;
        x.key[1] = 32 + lane < U ? __ldg(row + 32 + lane) : 0;
    };
    F32Query cur, nxt;
    fetch(q_lo + warp, cur);
#pragma unroll 1
    for (int i = q_lo + warp; i < q_hi; i += kF32Threads / 32) {
        fetch(i + kF32Threads / 32, nxt);
#pragma unroll
        for (int x = 0; x < 2; ++x)
            if ((unsigned)cur.key[x] >= (unsigned)L) { atomicOr(g.status, kStatusIdxClamped); cur.key[x] = cur.key[x] < 0 ? 0 : L - 1; }
        float s[NB];
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            float part[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {                      // (a sample behind the last reads row 0; its score is dropped)
                const int key = __shfl_sync(0xffffffffu, cur.key[n >> 1], (n & 1) * 16 + x * 4 + grp);
                float4 lo, hi;
                if (RESIDENT) { lo = Kl[key * 16 + at_lo]; hi = Kl[key * 16 + at_hi]; }
                else {
                    const float4 *kr = Kl + (long long)key * (k_pitch >> 2);
                    lo = __ldg(kr); hi = __ldg(kr + 1);
                }
                float2 p = make_float2(cur.q[0] * lo.x, cur.q[1] * lo.y);
                f32_fma2(p, cur.q[2], cur.q[3], lo.z, lo.w);
                f32_fma2(p, cur.q[4], cur.q[5], hi.x, hi.y);
                f32_fma2(p, cur.q[6], cur.q[7], hi.z, hi.w);
                part[x] = p.x + p.y;
            }
            const float r0 = (b0 ? part[2] : part[0]) + __shfl_xor_sync(0xffffffffu, b0 ? part[0] : part[2], 1);
            const float r1 = (b0 ? part[3] : part[1]) + __shfl_xor_sync(0xffffffffu, b0 ? part[1] : part[3], 1);
            float v = (b1 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, b1 ? r0 : r1, 2);
            v += __shfl_xor_sync(0xffffffffu, v, 4);
            s[n] = v;
        }
        float mx = -INFINITY, D = 0.f;
#pragma unroll
        for (int n = 0; n < NB; ++n)
            if (n * 16 + mine < U) mx = fmaxf(mx, s[n]);
#pragma unroll
        for (int o = 1; o <= 16; o <<= 1)
            if (o != 4) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));           // (lanes l and l ^ 4 hold the same scores)
#pragma unroll
        for (int n = 0; n < NB; ++n)
            if (n * 16 + mine < U) D += mx - s[n];
#pragma unroll
        for (int o = 1; o <= 16; o <<= 1)
            if (o != 4) D += __shfl_xor_sync(0xffffffffu, D, o);
        if (lane == 0) M_s[i] = U > 0 ? D * kScale / (float)U : 0.f;
        cur = nxt;
    }
}

template <bool RESIDENT>
__device__ __forceinline__ void f32_measure(const Geom &g, int unit, int b, int h, int L, int U, int q_lo, int q_hi,
                                            const float *__restrict__ Qu, const float *Ku, long long k_pitch,
                                            const int *__restrict__ sidx, float *M_s) {
    if (U <= 16) f32_measure_n<RESIDENT, 1>(g, unit, b, h, L, U, q_lo, q_hi, Qu, Ku, k_pitch, sidx, M_s);
    else if (U <= 32) f32_measure_n<RESIDENT, 2>(g, unit, b, h, L, U, q_lo, q_hi, Qu, Ku, k_pitch, sidx, M_s);
    else if (U <= 48) f32_measure_n<RESIDENT, 3>(g, unit, b, h, L, U, q_lo, q_hi, Qu, Ku, k_pitch, sidx, M_s);
    else f32_measure_n<RESIDENT, 4>(g, unit, b, h, L, U, q_lo, q_hi, Qu, Ku, k_pitch, sidx, M_s);
}

// Eight values per lane, reduced over the warp: lane l returns the result of value l >> 2 (the same in its four lanes).
template <class Op>
__device__ __forceinline__ float f32_reduce8(const float v[8], Op op) {
    const int lane = threadIdx.x & 31;
    float a[4], b[2];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const bool up = lane & 16;
        const float keep = up ? v[4 + x] : v[x], send = up ? v[x] : v[4 + x];
        a[x] = op(keep, __shfl_xor_sync(0xffffffffu, send, 16));
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const bool up = lane & 8;
        const float keep = up ? a[2 + x] : a[x], send = up ? a[x] : a[2 + x];
        b[x] = op(keep, __shfl_xor_sync(0xffffffffu, send, 8));
    }
    const bool up = lane & 4;
    float r = op(up ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4));
    r = op(r, __shfl_xor_sync(0xffffffffu, r, 2));
    return op(r, __shfl_xor_sync(0xffffffffu, r, 1));
}

// Rows of 256 bytes from global memory into shared memory, `n` of them (zeros from `valid` on), pitch in floats.
// `spread`: 16-byte piece c at c ^ (c >> 3) (see f32_measure).
__device__ __forceinline__ void f32_stage_rows(uint32_t dst, uint32_t pitch, const float *src, long long stride, int n, int valid,
                                               bool spread = false) {
#pragma unroll 4
    for (int e = threadIdx.x; e < n * 16; e += kF32Threads) {
        const int r = e >> 4, c = e & 15;
        const int at = spread ? c ^ (c >> 3) : c;
        const uint32_t d = dst + ((uint32_t)r * pitch + (uint32_t)at * 4u) * 4u;
        if (r < valid) cp_async_16(d, src + (long long)r * stride + c * 4);
        else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(d), "r"(0) : "memory");
    }
}

// The attention of the listed rows over the keys [lo, hi): on return P.m[0] / P.l hold the row states and the partial sums of the
// unnormalised rows lie at kF32OffP as [splits][rows][64]; returns splits.  Contains __syncthreads.
__device__ __forceinline__ int f32_attend(uint8_t *smem, const Geom &g, Fused32Persist &P, int b, int h, int L, int lo, int hi,
                                          int n_rows, int row_groups, const float *__restrict__ Qu,
                                          const float *__restrict__ Ku, const float *__restrict__ Vu) {
    const int tid = threadIdx.x, lane = tid & 31;
    float *Qs = reinterpret_cast<float *>(smem + kF32OffQ), *Ks = reinterpret_cast<float *>(smem + kF32OffK);
    float *Vs = reinterpret_cast<float *>(smem + kF32OffV), *Ps = reinterpret_cast<float *>(smem + kF32OffP);
    const int n_chunks = (hi - lo + kF32Chunk - 1) / kF32Chunk;
    auto stage_k = [&](int c) {
        const int k0 = lo + c * kF32Chunk;
        f32_stage_rows(smem_u32(Ks), kF32KPitch, Ku + (long long)k0 * g.ks[2], g.ks[2], kF32Chunk, hi - k0);
        cp_async_commit();
    };
    auto stage_v = [&](int c) {
        const int k0 = lo + c * kF32Chunk;
        f32_stage_rows(smem_u32(Vs), 64, Vu + (long long)k0 * g.vs[2], g.vs[2], kF32Chunk, hi - k0);
        cp_async_commit();
    };
#pragma unroll
    for (int e = tid; e < kF32MaxRows * 16; e += kF32Threads) {        // the listed rows; unused rows are zero
        const int r = e >> 4, c = e & 15, i = r < n_rows ? P.sel[r] : -1;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= 0 && i < L) v = __ldg(reinterpret_cast<const float4 *>(Qu + (long long)i * g.qs[2]) + c);
        reinterpret_cast<float4 *>(Qs)[e] = v;
    }
    if (tid < kF32MaxRows) { P.m[0][tid] = -INFINITY; P.l[tid] = 0.f; }
    if (n_chunks > 0) { stage_k(0); stage_v(0); }

    // scores: row group rg (8 rows), keys kg and kg + 64 of the chunk; values: row quad rq, columns 4 cq .., keys ks + splits * n
    const int kg = tid & 63, rg = tid >> 6;
    const int quads = 2 * row_groups, splits = kF32Threads / (16 * quads);
    const int cq = tid & 15, rq = (tid >> 4) % quads, ks = (tid >> 4) / quads;
    float2 o[4][2];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) o[x][y] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int c = 0; c < n_chunks; ++c) {
        const int valid = min(kF32Chunk, hi - lo - c * kF32Chunk);
        cp_async_wait<1>();                                    // K of this chunk (V may still be on its way)
        __syncthreads();
        float s[8][2];
        const bool lower = kg - lane < valid, upper = kg - lane + 64 < valid;  // of this warp's keys any exist (uniform)
        if (rg < row_groups) {
            const float4 *q = reinterpret_cast<const float4 *>(Qs + rg * 8 * 64);
            const float4 *k = reinterpret_cast<const float4 *>(Ks + kg * kF32KPitch);
            float2 e[8][2];                                    // sums over the even and the odd columns
#pragma unroll
            for (int x = 0; x < 8; ++x) e[x][0] = e[x][1] = make_float2(0.f, 0.f);
            if (upper) {                                       // both keys share the loads of the query rows
#pragma unroll 1
                for (int d = 0; d < 16; ++d) {
                    const float4 a0 = k[d], a1 = k[64 * kF32KPitch / 4 + d];
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const float4 v = q[x * 16 + d];
                        f32_fma2(e[x][0], v.x, v.y, a0.x, a0.y); f32_fma2(e[x][0], v.z, v.w, a0.z, a0.w);
                        f32_fma2(e[x][1], v.x, v.y, a1.x, a1.y); f32_fma2(e[x][1], v.z, v.w, a1.z, a1.w);
                    }
                }
            } else if (lower) {
#pragma unroll 2
                for (int d = 0; d < 16; ++d) {
                    const float4 a0 = k[d];
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const float4 v = q[x * 16 + d];
                        f32_fma2(e[x][0], v.x, v.y, a0.x, a0.y); f32_fma2(e[x][0], v.z, v.w, a0.z, a0.w);
                    }
                }
            }
#pragma unroll
            for (int x = 0; x < 8; ++x) { s[x][0] = e[x][0].x + e[x][0].y; s[x][1] = e[x][1].x + e[x][1].y; }
            float mx[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                s[x][0] = kg < valid ? s[x][0] * (kScale * kLog2e) : -INFINITY;
                s[x][1] = kg + 64 < valid ? s[x][1] * (kScale * kLog2e) : -INFINITY;
                mx[x] = fmaxf(s[x][0], s[x][1]);
            }
            const float r = f32_reduce8(mx, [](float a, float e) { return fmaxf(a, e); });
            if ((lane & 3) == 0) P.part[rg * 8 + (lane >> 2)][(tid >> 5) & 1] = r;
        }
        __syncthreads();
        if (c + 1 < n_chunks) stage_k(c + 1); else cp_async_commit();          // the K buffer is free
        // the new reference of a row, from what everyone can read; P.m of the next chunk is written beside it
        const float *m_old = P.m[c & 1];
        auto m_new = [&](int r) { return fmaxf(m_old[r], fmaxf(P.part[r][0], P.part[r][1])); };
        if (tid < row_groups * 8) P.m[(c + 1) & 1][tid] = m_new(tid);
        if (rg < row_groups) {
            float sum[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const float m = m_new(rg * 8 + x);
                s[x][0] = exp2f(s[x][0] - m); s[x][1] = exp2f(s[x][1] - m);
                sum[x] = s[x][0] + s[x][1];
            }
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                float4 *dst = reinterpret_cast<float4 *>(Ps + (kg + 64 * y) * kF32PPitch + rg * 8);
                dst[0] = make_float4(s[0][y], s[1][y], s[2][y], s[3][y]);
                dst[1] = make_float4(s[4][y], s[5][y], s[6][y], s[7][y]);
            }
            const float r = f32_reduce8(sum, [](float a, float e) { return a + e; });
            if ((lane & 3) == 0) P.sum[rg * 8 + (lane >> 2)][(tid >> 5) & 1] = r;
        }
        cp_async_wait<1>();                                    // V of this chunk
        __syncthreads();
        const float *m_cur = P.m[(c + 1) & 1];                 // alpha = exp2(old - new): 0 on the first chunk (m = -inf)
        if (tid < row_groups * 8) P.l[tid] = P.l[tid] * exp2f(m_old[tid] - m_cur[tid]) + (P.sum[tid][0] + P.sum[tid][1]);
        if (ks < splits) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float al = exp2f(m_old[rq * 4 + x] - m_cur[rq * 4 + x]);
#pragma unroll
                for (int y = 0; y < 2; ++y) { o[x][y].x *= al; o[x][y].y *= al; }
            }
#pragma unroll 4
            for (int k = ks; k < valid; k += splits) {
                const float4 p = *reinterpret_cast<const float4 *>(Ps + k * kF32PPitch + rq * 4), v = *reinterpret_cast<const float4 *>(Vs + k * 64 + cq * 4);
                const float pr[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int x = 0; x < 4; ++x) { f32_fma2(o[x][0], pr[x], pr[x], v.x, v.y); f32_fma2(o[x][1], pr[x], pr[x], v.z, v.w); }
            }
        }
        __syncthreads();
        if (c + 1 < n_chunks) stage_v(c + 1);                  // the V buffer is free
    }
    cp_async_wait<0>();
    __syncthreads();
    if ((n_chunks & 1) && tid < row_groups * 8) P.m[0][tid] = P.m[1][tid];
    if (ks < splits) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
            *reinterpret_cast<float4 *>(Ps + ((ks * quads + rq) * 4 + x) * 64 + cq * 4) = make_float4(o[x][0].x, o[x][0].y, o[x][1].x, o[x][1].y);
    }
    __syncthreads();
    return splits;
}

template <bool SPLIT>
__global__ void __launch_bounds__(kF32Threads, 1) k_forward_fused_fp32(
    Geom g, Fused32Args a, const float *__restrict__ Q, const float *__restrict__ K, const float *__restrict__ V,
    const int *__restrict__ sidx, float *__restrict__ O, int *__restrict__ sel_out, float *__restrict__ M_out) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x;
    float *M_s = reinterpret_cast<float *>(smem + a.off_persist);
    unsigned char *chosen = reinterpret_cast<unsigned char *>(M_s + a.m_floats);
    Fused32Persist &P = *reinterpret_cast<Fused32Persist *>(smem + a.off_persist + f32_arrays_bytes(a.m_floats, g.T));
    const int split = SPLIT ? a.split : 1, part = SPLIT ? (int)(blockIdx.x % split) : 0;
    if (SPLIT) cluster_arrive();                                // this CTA runs: its shared memory may be written to
    pdl_enter();
    int b = (int)(blockIdx.x / split) / g.H;
    const int h = (int)(blockIdx.x / split) % g.H;
    if (!SPLIT && a.by_length) {                                // longest sequences first, as in k_forward_fused
        b = sequence_of_rank(g, b, kF32Threads, &P.b_ranked);
    }
    const int unit = b * g.H + h;
    const int L = seq_len(g, b);
    const int U = min(g.U_tab[L], g.idx_cols);
    const int u = min(min(g.u_tab[L], g.u_max), L);
    const bool given = a.sel_in != nullptr;                    // steps (d)+(e) only, for a given index set
    const float *Qu = Q + unit_off(g.qs, b, h), *Ku = K + unit_off(g.ks, b, h), *Vu = V + unit_off(g.vs, b, h);
    for (int i = tid; i < g.T; i += kF32Threads) { chosen[i] = 0; if (i >= L && !given) M_s[i] = 0.f; }

    phase_stamp(g, 0);
    // ---- steps (a)+(b): every CTA of the unit a range of the queries; its values go to the others -----------------
    if (SPLIT) cluster_wait();                                  // every CTA of the unit runs
    if (L > 0 && !given) {
        const int per = (L + split - 1) / split;
        const int q_lo = min(part * per, L), q_hi = min(q_lo + per, L);
        if (a.resident) {
            f32_stage_rows(smem_u32(smem), 64, Ku, g.ks[2], L, L, true);
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
            phase_stamp(g, 1);                                 // the keys have landed
            f32_measure<true>(g, unit, b, h, L, U, q_lo, q_hi, Qu, reinterpret_cast<const float *>(smem), 64, sidx, M_s);
        } else {
            f32_measure<false>(g, unit, b, h, L, U, q_lo, q_hi, Qu, Ku, g.ks[2], sidx, M_s);
        }
        __syncthreads();
        if (SPLIT) {
            for (int x = 1; x < split; ++x) {
                const uint32_t dst = peer_addr(smem_u32(M_s), part + x < split ? part + x : part + x - split);
                for (int i = q_lo + tid; i < q_hi; i += kF32Threads) peer_store(dst + 4u * (uint32_t)i, M_s[i]);
            }
            cluster_arrive();
            cluster_wait();
        }
    }
    __syncthreads();
    phase_stamp(g, 2);                                         // steps (a)+(b) done
    if (M_out != nullptr && !given && part == 0)
        for (int i = tid; i < g.T; i += kF32Threads) M_out[(long long)unit * g.T + i] = M_s[i];

    // ---- step (c) -----------------------------------------------------------------------------
    const int n_rows = given ? g.u_max : u;                    // a given list is taken at its full width
    if (!given) {
        block_select_short<3>([&](int i) { return float_key(M_s[i]); }, L, u, kF32MaxRows, P.sel, P.select, kF32Threads, 0);
        for (int r = tid; r < g.u_max; r += kF32Threads) {
            const int i = r < kF32MaxRows ? P.sel[r] : -1;
            if (part == 0) sel_out[(long long)unit * g.u_max + r] = i;
            if (i >= 0) chosen[i] = 1;
        }
    } else {
        for (int r = tid; r < kF32MaxRows; r += kF32Threads) {
            const int i = r < g.u_max ? a.sel_in[(long long)unit * g.u_max + r] : -1;
            P.sel[r] = (i >= 0 && i < L) ? i : -1;              // entries outside the sequence are ignored
            if (i >= 0 && i < L) chosen[i] = 1;
        }
    }
    __syncthreads();
    phase_stamp(g, 3);                                         // step (c) done

    // ---- step (d), with the column sums of V as one more row ------------------------------------------------
    if (L > 0) {
        const int sum_row = a.own_v ? -1 : n_rows;
        const int row_groups = (max(n_rows, sum_row + 1) + 7) / 8;
        const int per = SPLIT ? (L + split - 1) / split : L;
        const int lo = min(part * per, L), hi = min(lo + per, L);
        const int splits = f32_attend(smem, g, P, b, h, L, lo, hi, n_rows, row_groups, Qu, Ku, Vu);
        phase_stamp(g, 6);                                     // step (d): the merge is left
        const float *Ps = reinterpret_cast<const float *>(smem + kF32OffP);
        const int row = tid >> 3, c8 = tid & 7;
        float acc[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) acc[x] = 0.f;
        if (row < row_groups * 8)
            for (int s = 0; s < splits; ++s) {
                const float4 *src = reinterpret_cast<const float4 *>(Ps + (s * row_groups * 8 + row) * 64 + c8 * 8);
                const float4 x = src[0], y = src[1];
                acc[0] += x.x; acc[1] += x.y; acc[2] += x.z; acc[3] += x.w;
                acc[4] += y.x; acc[5] += y.y; acc[6] += y.z; acc[7] += y.w;
            }
        if (SPLIT) {
            // as in k_forward_fused: the states of every CTA's key range stay in its shared memory, CTA p finishes the rows
            // r = p (mod split), and each CTA the fill row
            float *mine = reinterpret_cast<float *>(smem + kF32OffV);
            if (row < row_groups * 8) {
                float *dst = mine + row * 66;
                if (c8 == 0) { dst[0] = P.m[0][row]; dst[1] = P.l[row]; }
#pragma unroll
                for (int x = 0; x < 8; x += 2) *reinterpret_cast<float2 *>(dst + 2 + 8 * c8 + x) = make_float2(acc[x], acc[x + 1]);
            }
            cluster_arrive();
            cluster_wait();
            const int c = tid & 63;
            for (int k = tid >> 6; k == 0 || part + (k - 1) * split < n_rows; k += kF32Threads / 64) {   // 0: the fill row
                const int r = k == 0 ? sum_row : part + (k - 1) * split;
                const int i = k == 0 ? 0 : P.sel[r];
                if (r < 0 || i < 0) continue;
                const float v = merge_states(split, smem_u32(mine), r, c);
                if (k == 0) P.vbar[c] = v;
                else O[unit_off(g.os, b, h) + (long long)i * g.os[2] + c] = v;
            }
            cluster_arrive();                                   // done with the other CTAs' memory (awaited before the exit)
        } else {
            const float l = row < row_groups * 8 ? P.l[row] : 0.f, inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
            for (int x = 0; x < 8; ++x) acc[x] *= inv;
            if (row < n_rows) {
                const int i = P.sel[row];
                if (i >= 0) store8(O + unit_off(g.os, b, h) + (long long)i * g.os[2], c8, acc);
            } else if (row == sum_row) {
#pragma unroll
                for (int x = 0; x < 8; ++x) P.vbar[8 * c8 + x] = acc[x];
            }
        }
    }
    __syncthreads();
    phase_stamp(g, 4);                                         // step (d) done

    // ---- step (e) -----------------------------------------------------------------------------
    {
        const int sub = tid & 7, per = (g.T + split - 1) / split;
        float fillv[8], zero8[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) { fillv[t] = (L > 0 && !a.own_v) ? P.vbar[sub * 8 + t] : 0.f; zero8[t] = 0.f; }
        float *Ou = O + unit_off(g.os, b, h);
        for (int i = part * per + (tid >> 3); i < min(g.T, (part + 1) * per); i += kF32Threads / 8) {
            float *dst = Ou + (long long)i * g.os[2];
            if (i >= L) store8(dst, sub, zero8);
            else if (chosen[i]) continue;
            else if (a.own_v) { float v[8]; load8(Vu + (long long)i * g.vs[2], sub, v); store8(dst, sub, v); }
            else store8(dst, sub, fillv);
        }
    }
    __syncthreads();
    phase_stamp(g, 5);                                         // step (e) done
    if (SPLIT && L > 0) cluster_wait();                        // nobody reads this CTA's states any more
}

// CTAs per unit: as many (up to 8) as leave every cluster resident at once; see fused_split in psattn_fused.cu.  us per call with
// 1 / 2 / 4 / 8 CTAs per unit: B1 H4 T64 14.4 / 14.1 / 12.8 / 13.0, T128 21.4 / 17.7 / 14.6 / 13.9, T200 32.0 / 21.9 / 17.1 / 15.1.
static int f32_split(const Geom &g) {
    static ClusterRecord clusters;
    const int units = g.B * g.H;
    if (g.T < 48) return 1;
    for (int split = kMaxSplit; split > 1; --split)
        if (units <= max_clusters(k_forward_fused_fp32<true>, clusters, split, kF32Threads, kF32MaxSmem)) return split;
    return 1;
}

// cudaErrorNotSupported: more than 63 selected rows or 64 samples, sequences too long for the selection's registers, or
// sample lists shared by the queries (the caller runs the staged schedule).
cudaError_t launch_forward_fused_fp32(const Geom &g, int U_max, int own_v, const void *Q, const void *K, const void *V,
                                      const int *sidx, void *O, int *sel, float *M_out, const int *sel_in, cudaStream_t st) {
    if (g.B * g.H == 0) return cudaSuccess;
    const bool given = sel_in != nullptr;
    if (g.u_max > kF32MaxRows - 1) return cudaErrorNotSupported;
    if (!given && (U_max > 64 || U_max < 1 || g.idx_shared || g.T > 3 * kF32Threads)) return cudaErrorNotSupported;
    Fused32Args a;
    a.m_floats = given ? 0 : g.T;
    const size_t tail = f32_arrays_bytes(a.m_floats, g.T) + sizeof(Fused32Persist) + 128;
    const size_t keys = (size_t)g.T * 256;
    a.resident = !given && keys + tail <= kF32MaxSmem;
    const size_t phase = a.resident && keys > kF32AttendBytes ? keys : kF32AttendBytes;
    a.off_persist = (uint32_t)((phase + 127) / 128 * 128);
    const size_t smem = a.off_persist + tail;
    if (smem > kF32MaxSmem) return cudaErrorNotSupported;
    a.own_v = own_v;
    a.sel_in = sel_in;
    static SmemGrant grant, grant_split;
    if (cudaError_t e = grant_dynamic_smem(k_forward_fused_fp32<false>, grant, kF32MaxSmem)) return e;
    if (cudaError_t e = grant_dynamic_smem(k_forward_fused_fp32<true>, grant_split, kF32MaxSmem)) return e;
    a.split = f32_split(g);
    a.by_length = g.lengths != nullptr && g.B * g.H > device_sm_count() && g.B <= 256;
    cudaError_t e = launch_split(a.split > 1 ? k_forward_fused_fp32<true> : k_forward_fused_fp32<false>, (unsigned)(g.B * g.H),
                                 a.split, kF32Threads, smem, st, g, a, (const float *)Q, (const float *)K, (const float *)V,
                                 sidx, (float *)O, sel, M_out);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace psattn
