// Stand-alone kernel around attend_rows_run: step (d) for row lists of at most 64 rows per unit
// (the selected queries of the sparse path).  One CTA = (unit, key split).
#include "psattn_attend_rows.cuh"
#include "psattn_launch.h"

namespace psattn {

using namespace sm100;

struct Attend64Args {
    const int *rows;            // [unit][rows_stride]
    int n_rows, rows_stride;
    int n_splits, split_keys;   // split_keys is a multiple of 256
    float *part_ml, *part_acc;
    void *out;
    long long out_unit_stride, out_row_stride;
    int out_by_position, out_fp32;
    int pos_t, pos_h, pos_b;
    float *vbar;                // if non-null: mean(V) [unit][64], from an extra all-weights-1 row (slot n_rows)
};

__global__ void __launch_bounds__(ArWide::kThreads, 1) k_attend64(Geom g, Attend64Args a, const __nv_bfloat16 *__restrict__ Q,
                                                            const __grid_constant__ CUtensorMap tmK,
                                                            const __grid_constant__ CUtensorMap tmV) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x;
    const int split = blockIdx.x, unit = blockIdx.y;
    if ((smem_u32(smem) & 1023u) != 0u) {                      // swizzled tiles need a 1024-byte base
        if (tid == 0) atomicOr(g.status, kStatusWaitExpired);
        return;
    }
    if (tid == 32) { tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); }
    pdl_enter();
    KernelSpan span(g, kKernelAttend64);

    AttendRowsJob j;
    j.b = unit / g.H; j.h = unit % g.H; j.L = seq_len(g, j.b);
    j.lo = min(j.L, split * a.split_keys); j.hi = min(j.L, j.lo + a.split_keys);
    j.rows = a.rows + (long long)unit * a.rows_stride; j.n_rows = a.n_rows;
    j.pos_t = a.pos_t; j.pos_h = a.pos_h; j.pos_b = a.pos_b;
    j.sum_row = a.vbar ? a.n_rows : -1;
    if (tid == ArWide::kLoader) attend_rows_start<ArWide>(smem, g, j, &tmK, &tmV, 1);
    float m_rows[1], l_rows[1], acc_rows[1][8];
    if (!attend_rows_run<ArWide>(smem, g, j, Q, &tmK, &tmV, 1, m_rows, l_rows, acc_rows)) return;
    const float m_run = m_rows[0], l_run = l_rows[0];
    float (&acc)[8] = acc_rows[0];

    const int r = tid >> 3, c8 = tid & 7;
    const int n_slots = a.n_rows + (a.vbar ? 1 : 0);               // row slots per unit in the split partials
    if (r >= n_slots) return;
    const bool sums = r == j.sum_row;                              // column sums of V over [lo, hi), l = key count
    const int i = sums ? 0 : j.rows[r];
    const bool row_ok = sums || (i >= 0 && i < j.L);
    if (a.n_splits > 1) {
        const long long slot = ((long long)unit * n_slots + r) * a.n_splits + split;
        if (c8 == 0) {
            a.part_ml[2 * slot] = row_ok && l_run > 0.f ? m_run : -INFINITY;
            a.part_ml[2 * slot + 1] = row_ok ? l_run : 0.f;
        }
        store8(a.part_acc + slot * kD, c8, acc);
        return;
    }
    const float inv = row_ok && l_run > 0.f ? 1.f / l_run : 0.f;
#pragma unroll
    for (int x = 0; x < 8; ++x) acc[x] = row_ok ? acc[x] * inv : 0.f;
    if (sums) {
        store8(a.vbar + (long long)unit * kD, c8, acc);
    } else if (a.out_by_position) {
        if (row_ok) store8(reinterpret_cast<__nv_bfloat16 *>(a.out) + unit_off(g.os, j.b, j.h) + (long long)i * g.os[2], c8, acc);
    } else if (a.out_fp32) {
        store8(reinterpret_cast<float *>(a.out) + (long long)unit * a.out_unit_stride + (long long)r * a.out_row_stride, c8, acc);
    } else {
        store8(reinterpret_cast<__nv_bfloat16 *>(a.out) + (long long)unit * a.out_unit_stride + (long long)r * a.out_row_stride, c8, acc);
    }
}

bool make_rows_map(CUtensorMap *map, const void *base, const Geom &g, const long long s[3], int box_rows,
                   int swizzle128, int pos[3]);

// Host-side check with no side effect: would launch_attend64 take this call?
bool attend64_supported(const Geom &g, const void *K, const void *V, int n_rows, int with_vbar) {
    if (n_rows + (with_vbar ? 1 : 0) > kArMaxRows) return false;
    CUtensorMap tmK, tmV;
    int posK[3], posV[3];
    if (!make_rows_map(&tmK, K, g, g.ks, 128, 1, posK) || !make_rows_map(&tmV, V, g, g.vs, 128, 1, posV)) return false;
    return posK[0] == posV[0] && posK[1] == posV[1] && posK[2] == posV[2];
}

// cudaErrorNotSupported: more than 64 rows (63 with vbar), no row list, or no tensor map for the layout.
cudaError_t launch_attend64(const Geom &g, const void *Q, const void *K, const void *V, const int *rows,
                            int n_rows, int rows_stride, int n_splits, int split_keys, float *part_ml,
                            float *part_acc, void *out, long long out_unit_stride, long long out_row_stride,
                            int out_by_position, int out_fp32, float *vbar, cudaStream_t st) {
    if (g.B * g.H == 0 || n_rows == 0) return cudaSuccess;
    if (n_rows + (vbar ? 1 : 0) > kArMaxRows || rows == nullptr || (split_keys % 256) != 0) return cudaErrorNotSupported;
    if ((long long)g.B * g.H > 65535) return cudaErrorNotSupported;         // the unit index is gridDim.y
    Attend64Args a;
    a.rows = rows; a.n_rows = n_rows; a.rows_stride = rows_stride;
    a.n_splits = n_splits; a.split_keys = split_keys;
    a.part_ml = part_ml; a.part_acc = part_acc; a.out = out;
    a.out_unit_stride = out_unit_stride; a.out_row_stride = out_row_stride;
    a.out_by_position = out_by_position; a.out_fp32 = out_fp32; a.vbar = vbar;
    CUtensorMap tmK, tmV;
    int posK[3], posV[3];
    if (!make_rows_map(&tmK, K, g, g.ks, 128, 1, posK) || !make_rows_map(&tmV, V, g, g.vs, 128, 1, posV))
        return cudaErrorNotSupported;
    if (posK[0] != posV[0] || posK[1] != posV[1] || posK[2] != posV[2]) return cudaErrorNotSupported;
    a.pos_t = posK[0]; a.pos_h = posK[1]; a.pos_b = posK[2];
    static SmemGrant grant;
    if (cudaError_t e = grant_dynamic_smem(k_attend64, grant, ArWide::kBytes)) return e;
    dim3 grid((unsigned)n_splits, (unsigned)(g.B * g.H));
    cudaError_t le = launch_pdl(k_attend64, grid, dim3(ArWide::kThreads), ArWide::kBytes, st, g, a, (const __nv_bfloat16 *)Q, tmK, tmV);
    if (le != cudaSuccess) { note_launch(); return le; }
    note_launch();
    return cudaGetLastError();
}

}  // namespace psattn
