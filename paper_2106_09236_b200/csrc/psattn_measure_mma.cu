// Stand-alone kernel around measure_resident: steps (a)+(b) (Eq. 11) for bf16 inputs.
// One CTA = (unit, slice of its queries).
#include "psattn_launch.h"
#include "psattn_measure_mma.cuh"
#include "psattn_measure_stream.cuh"

namespace psattn {

using namespace sm100;

constexpr int kMeasureThreads = 640;

struct MeasureMmaArgs {
    int q_slices;               // CTAs per unit
    int pos_t, pos_h, pos_b;    // TMA coordinate slots of t, h, b
    uint32_t stage_bytes;       // bytes of one staging buffer (Q tile + sample tile)
    uint32_t k_bytes;           // bytes reserved for the resident keys
};

__global__ void __launch_bounds__(kMeasureThreads, 1) k_measure_mma(Geom g, MeasureMmaArgs a,
                                                                    const __nv_bfloat16 *__restrict__ Q,
                                                                    const int *__restrict__ sidx,
                                                                    float *__restrict__ M,
                                                                    const __grid_constant__ CUtensorMap tmK) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t bar;
    const int tid = threadIdx.x;
    const int unit = blockIdx.x / a.q_slices, slice = blockIdx.x % a.q_slices;
    const int b = unit / g.H, h = unit % g.H;
    const int L = seq_len(g, b);
    const int U = min(g.U_tab[L], g.idx_cols);
    const int per = (g.T + a.q_slices - 1) / a.q_slices;
    const int q_lo = slice * per, q_hi = min(g.T, q_lo + per);
    const int q_end = min(q_hi, L);
    float *Mu = M + (long long)unit * g.T;

    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
        if (q_lo < L) measure_issue_keys(smem, &bar, &tmK, L, b, h, a.pos_t, a.pos_h);
    }
    // rows of padded queries are zero
    for (int i = max(q_lo, L) + tid; i < q_hi; i += kMeasureThreads) Mu[i] = 0.f;
    __syncthreads();
    if (L == 0 || q_lo >= L) return;
    measure_resident<kMeasureThreads>(smem, &bar, 0u, a.k_bytes, a.stage_bytes, g, unit, b, h, L, U, q_lo, q_end, Q,
                                      sidx, Mu);
}

// Streaming form (keys gathered from L2 through per-warp rings): any T_max.
constexpr int kStreamThreads = 768;      // at most: fewer warps where long sample rows leave no room for their buffers

__global__ void __launch_bounds__(kStreamThreads, 1) k_measure_stream(Geom g, uint32_t warp_stage_bytes,
                                                                      const __nv_bfloat16 *__restrict__ Q,
                                                                      const __nv_bfloat16 *__restrict__ K,
                                                                      const int *__restrict__ sidx, float *__restrict__ M) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ unsigned long long warp_sum[kStreamThreads / 32];
    const int n_threads = blockDim.x, n_warps = n_threads >> 5;
    // shared memory: rings, staging buffers, weight of all groups of the sequences before b (b = 0 .. B)
    unsigned long long *before = reinterpret_cast<unsigned long long *>(smem + n_warps * (kStreamRing * kStreamRoundBytes + 2 * warp_stage_bytes));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_enter();
    KernelSpan span(g, kKernelMeasure);
    // weights of the sequences, added up in order (thread t takes sequences t * per ..)
    {
        const int per = (g.B + n_threads - 1) / n_threads;
        auto weight_of = [&](int b) {
            const int L = seq_len(g, b);
            return L > 0 ? (unsigned long long)stream_groups(L) * g.H * stream_weight(min(g.U_tab[L], g.idx_cols)) : 0ull;
        };
        unsigned long long mine = 0;
        for (int b = tid * per; b < min(g.B, (tid + 1) * per); ++b) mine += weight_of(b);
        unsigned long long incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        unsigned long long at = incl - mine;
        for (int w = 0; w < warp; ++w) at += warp_sum[w];
        for (int b = tid * per; b < min(g.B, (tid + 1) * per); ++b) { before[b] = at; at += weight_of(b); }
        if (tid == 0) {
            unsigned long long all = 0;
            for (int w = 0; w < n_warps; ++w) all += warp_sum[w];
            before[g.B] = all;
        }
        __syncthreads();
    }
    const unsigned long long all = before[g.B];
    const unsigned long long w_lo = all * blockIdx.x / gridDim.x, w_hi = all * (blockIdx.x + 1) / gridDim.x;
    // zeros at padded positions, unit by unit
    for (int unit = blockIdx.x; unit < g.B * g.H; unit += gridDim.x)
        for (int i = seq_len(g, unit / g.H) + tid; i < g.T; i += n_threads) M[(long long)unit * g.T + i] = 0.f;

    // this warp's groups: every n_warps-th of the CTA's range
    int b = 0;
    for (int step = kStreamMaxB / 2; step > 0; step >>= 1)                 // last sequence that starts at or before w_lo
        if (b + step < g.B && before[b + step] <= w_lo) b += step;
    struct Group { int b, h, i0, rows, L, U; };
    int k = 0, k_hi = 0, skip = warp;                          // within sequence b: next group number, end; groups to skip first
    bool open = false;
    auto next = [&](Group &x) {                                // false: no more groups
        for (; b < g.B && before[b] < w_hi; ++b, open = false) {
            const int L = seq_len(g, b);
            if (L == 0) continue;
            const int ng = stream_groups(L), U = min(g.U_tab[L], g.idx_cols);
            if (!open) {
                stream_range(before[b], ng * g.H, stream_weight(U), w_lo, w_hi, k, k_hi);
                open = true;
            }
            if (k + skip >= k_hi) { skip -= max(0, k_hi - k); continue; }
            k += skip; skip = 0;
            x.b = b; x.h = k / ng; x.i0 = (k - x.h * ng) * 8; x.rows = min(8, L - x.i0); x.L = L; x.U = U;
            ++k; skip = n_warps - 1;
            return true;
        }
        return false;
    };
    StreamCtx cx;
    cx.ring = smem_u32(smem) + (uint32_t)warp * kStreamRing * kStreamRoundBytes;
    cx.idx_pitch = measure_idx_pitch(g.idx_cols); cx.status = g.status; cx.k_row_bytes = (uint32_t)(g.ks[2] * 2);
    const uint32_t stage0 = smem_u32(smem) + n_warps * kStreamRing * kStreamRoundBytes + (uint32_t)warp * 2u * warp_stage_bytes;
    // Q rows, then sample rows, of a group into one of the warp's two buffers; nobody else reads them, so the warps never meet at
    // a barrier and drift apart: the pipeline bubble at the start of a group does not hit all of them at once
    auto stage = [&](const Group &x, int buf) {
        const uint32_t dst = stage0 + (uint32_t)buf * warp_stage_bytes;
        const __nv_bfloat16 *Qu = Q + unit_off(g.qs, x.b, x.h);
        for (int e = lane; e < x.rows * 8; e += 32)
            cp_async_16(dst + (uint32_t)e * 16u, Qu + (long long)(x.i0 + (e >> 3)) * g.qs[2] + (e & 7) * 8);
        measure_stage_samples(dst + 1024u, sidx + ((g.idx_per_head ? (long long)(x.b * g.H + x.h) : (long long)x.b) * g.T + x.i0) * g.idx_cols,
                              x.rows, g.idx_cols);
        cp_async_commit();
    };
    Group cur, nxt;
    bool have = next(cur);
    if (have) stage(cur, 0);
    for (int n = 0; have; ++n) {
        cp_async_wait<0>();                                    // this lane's part of the group (nothing else is pending)
        __syncwarp();
        asm volatile("mov.u32 %0, %1;" : "=r"(cx.epoch0) : "r"(n << 8) : "memory");
        have = next(nxt);
        if (have) stage(nxt, (n + 1) & 1);                     // lands while this group is worked on
        cx.q_tile = stage0 + (uint32_t)(n & 1) * warp_stage_bytes;
        cx.idx_tile = cx.q_tile + 1024u;
        cx.rows = cur.rows; cx.L = cur.L; cx.U = min(cur.U, kMeasureMaxU);
        cx.Ku = K + unit_off(g.ks, cur.b, cur.h);
        cx.out = M + (long long)(cur.b * g.H + cur.h) * g.T + cur.i0;
        measure_stream_group(cx);
        __syncwarp();                                          // the group's buffer may be staged again from now on
        cur = nxt;
    }
    cp_async_wait<0>();
}

// ---- host side ----------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn2)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

bool make_rows_map(CUtensorMap *map, const void *base, const Geom &g, const long long s[3], int box_rows,
                   int swizzle128, int pos[3]) {
    static const EncodeTiledFn2 enc = reinterpret_cast<EncodeTiledFn2>(tensor_map_encoder());
    if (!enc) return false;
    struct Dim { long long size, stride; int which; } dims[3] = {{g.T, s[2], 0}, {g.H, s[1], 1}, {g.B, s[0], 2}};
    for (int x = 0; x < 3; ++x)
        for (int y = x + 1; y < 3; ++y)
            if (dims[y].stride < dims[x].stride) { Dim tmp = dims[x]; dims[x] = dims[y]; dims[y] = tmp; }
    cuuint64_t gdim[4] = {(cuuint64_t)kD, 0, 0, 0};
    cuuint64_t gstr[3];
    cuuint32_t box[4] = {(cuuint32_t)kD, 1, 1, 1}, estr[4] = {1, 1, 1, 1};
    for (int x = 0; x < 3; ++x) {
        if (dims[x].stride <= 0) return false;
        gdim[x + 1] = (cuuint64_t)dims[x].size;
        gstr[x] = (cuuint64_t)dims[x].stride * 2;
        pos[dims[x].which] = x + 1;
        if (dims[x].which == 0) box[x + 1] = (cuuint32_t)box_rows;
    }
    CUresult rc = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), gdim, gstr, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE,
                      swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS;
}

// cudaErrorNotSupported: T_max too long for resident keys, U above four rounds, or no tensor map.
cudaError_t launch_measure_mma(const Geom &g, int U_max, const void *Q, const void *K, const int *sidx, float *M,
                               cudaStream_t st) {
    if (g.B * g.H == 0) return cudaSuccess;
    const size_t k_bytes = measure_k_bytes(g.T);
    const size_t stage_bytes = measure_stage_bytes(kMeasureThreads, g.idx_cols);
    const size_t smem = k_bytes + kMeasureStages * stage_bytes;
    if (smem > 225 * 1024 || U_max > kMeasureMaxU || U_max < 1) return cudaErrorNotSupported;
    CUtensorMap tmK;
    int pos[3];
    if (!make_rows_map(&tmK, K, g, g.ks, kMeasureBoxRows, 0, pos)) return cudaErrorNotSupported;
    MeasureMmaArgs a;
    a.pos_t = pos[0]; a.pos_h = pos[1]; a.pos_b = pos[2];
    a.stage_bytes = (uint32_t)stage_bytes; a.k_bytes = (uint32_t)k_bytes;
    const int units = g.B * g.H;
    // resident CTAs per SM by shared memory; slices so that the grid covers the SMs
    const int per_sm = smem <= 100 * 1024 ? 2 : 1;
    int slices = (device_sm_count() * per_sm) / units;
    if (slices < 1) slices = 1;
    if (slices > 8) slices = 8;
    a.q_slices = slices;
    static SmemGrant grant;
    if (cudaError_t e = grant_dynamic_smem(k_measure_mma, grant, smem)) return e;
    k_measure_mma<<<(unsigned)(units * slices), kMeasureThreads, smem, st>>>(g, a, (const __nv_bfloat16 *)Q, sidx, M, tmK);
    note_launch();
    return cudaGetLastError();
}

}  // namespace psattn

namespace psattn {

// cudaErrorNotSupported: more than 64 samples per query, sample rows too wide for shared memory, or key rows of a unit
// spread over 4 GB or more.
cudaError_t launch_measure_stream(const Geom &g, int U_max, const void *Q, const void *K, const int *sidx, float *M,
                                  cudaStream_t st) {
    if (g.B * g.H == 0) return cudaSuccess;
    if (U_max > kMeasureMaxU || U_max < 1) return cudaErrorNotSupported;
    if (g.ks[2] <= 0 || (long long)g.T * g.ks[2] * 2 >= (1ll << 32)) return cudaErrorNotSupported;
    const size_t warp_stage = (1024 + (size_t)8 * measure_idx_pitch(g.idx_cols) * 4 + 15) / 16 * 16;
    const size_t table = ((size_t)(g.B < kStreamMaxB ? g.B : kStreamMaxB) + 1) * 8;
    const size_t per_warp = kStreamRing * kStreamRoundBytes + 2 * warp_stage, room = 226 * 1024 - table;
    int warps = (int)(room / per_warp);
    if (warps > kStreamThreads / 32) warps = kStreamThreads / 32;
    if (warps < 8) return cudaErrorNotSupported;               // sample rows of hundreds of columns: the plain kernel
    const size_t smem = (size_t)warps * per_warp + table;
    static SmemGrant grant;
    if (cudaError_t e = grant_dynamic_smem(k_measure_stream, grant, smem)) return e;
    for (int b0 = 0; b0 < g.B; b0 += kStreamMaxB) {
        Geom part = g;
        part.B = g.B - b0 < kStreamMaxB ? g.B - b0 : kStreamMaxB;
        if (g.lengths) part.lengths = g.lengths + b0;
        const long long idx_b = (long long)(g.idx_per_head ? g.H : 1) * g.T * g.idx_cols;
        cudaError_t e = launch_pdl(k_measure_stream, dim3((unsigned)device_sm_count()), dim3((unsigned)warps * 32), smem, st, part,
                                   (uint32_t)warp_stage, (const __nv_bfloat16 *)Q + b0 * g.qs[0], (const __nv_bfloat16 *)K + b0 * g.ks[0],
                                   sidx + b0 * idx_b, M + (long long)b0 * g.H * g.T);
        note_launch();
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace psattn
