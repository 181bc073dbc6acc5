// Step (d) (Eq. 7-8) for up to 64 listed rows of one unit, as a routine of a CTA of 512 (or 256) threads on mma.sync.
//
// The step is short and its operands are thin (u <= 64 rows), so what it costs is the chain of dependent steps, not
// the tensor pipe: on tcgen05 every key tile went TMA -> product -> TMEM -> registers -> shared memory -> product ->
// TMEM -> registers with a barrier between any two, 6.9 us for a single tile and 9.1 us for T = 1024, while the M = 64
// products kept the pipe a few per cent busy.  Here scores and weights stay in the registers of one warp from the first
// product to the second, and no warp waits for another before the merge at the end.
//
//   K and V stream in chunks of 256 (128) keys by TMA (128-byte swizzle) through a ring of three (two) stages; a chunk's stage is
//   refilled by whichever warp is the last to leave it.
//   A warp owns one tile of 16 rows and one key group: the blocks of 32 keys whose number is the group's modulo the
//   number of groups, so that short sequences spread over all warps as well.  Groups: 16, 8, 5 or 4 for one to four
//   row tiles (fewer row tiles leave more warps to the keys).
//   S = Q K^T (mma.m16n8k16, K through ldmatrix), softmax in the registers (base 2) against a reference per row that
//   moves only when a score exceeds it by more than 8, P as bf16 straight into the A operand of O += P V (V through
//   ldmatrix.trans).
//   At the end the groups' states (m, l, O) are merged through shared memory, in group order.
// Bound: instruction issue, then mma.sync (one m16n8k16 per 8 clocks and scheduler, measured): a trip of a warp over 32
// keys is 32 products, 16 ldmatrix and about 110 other instructions; four warps of a scheduler take 1520 clocks per trip each,
// of which the products are 1100.  With three row tiles T = 1024 takes 7.0 us, T = 512 3.8 us, one tile of keys 1.3 us.
// A row whose query is zero gets the weight exp2(0) = 1 on every key: its O is the column sum of V and its l the number
// of keys, which is how mean(V) comes out of the same pass.
#pragma once
#include "psattn_common.cuh"
#include "psattn_measure_mma.cuh"
#include "psattn_sm100.cuh"

namespace psattn {

constexpr int kArMaxRows = 64;
constexpr int kArBlock = 32;                                 // keys per trip of a warp
constexpr uint32_t kArTile = 16384;                          // one 128-key K or V tile
constexpr uint32_t kArOffQ = 0;                              // 64 rows x 128 B
constexpr uint32_t kArOffStage = 8192;                       // per stage: K tiles, then V tiles
// Shape of the CTA: threads, keys per stage, stages of the ring.
template <int THREADS, int CHUNK, int STAGES>
struct AttendRowsShape {
    static constexpr int kThreads = THREADS, kChunk = CHUNK, kStages = STAGES;
    static constexpr int kLoader = THREADS - 32;             // the thread that starts the copies of the first stages
    static constexpr int kPerChunk = CHUNK / kArBlock;
    static constexpr int kRows = kArMaxRows * 8 / THREADS;   // rows per thread of the result
    static constexpr uint32_t kOffV = CHUNK * 128, kStageBytes = 2 * kOffV;
    static constexpr uint32_t kOffBar = kArOffStage + STAGES * kStageBytes;
    static constexpr uint32_t kBytes = kOffBar + 128;
};
typedef AttendRowsShape<512, 256, 3> ArWide;                 // alone on its SM
typedef AttendRowsShape<256, 128, 2> ArHalf;                 // two CTAs per SM
constexpr int kArMostStages = 3;
constexpr int kArPitch = 72;                                 // floats per row of the merge buffer: O[64], m, l

struct AttendRowsJob {
    int b, h, L;                 // unit and its valid length
    int lo, hi;                  // key range of this CTA
    const int *rows;             // listed positions (global or shared), or null = identity
    int n_rows;                  // <= 64
    int pos_t, pos_h, pos_b;     // TMA coordinate slots
    int sum_row;                 // slot (>= n_rows, < 64) with a zero query although it lists none; -1 = none
};

struct AttendRowsBars {
    uint64_t full[kArMostStages];
    int left[kArMostStages];         // warps that have left the stage
    int issued[kArMostStages];       // copies started into the stage
    int abort_flag;
};

// One thread: the TMA copies of chunk c.  (The test hook makes the last chunk wait for more bytes than are sent: with more
// chunks than stages that is a refilled stage, and the copies of other stages are in flight when the wait runs out.)
template <class S>
__device__ __forceinline__ void attend_rows_load(uint8_t *smem, const Geom &g, const AttendRowsJob &j, const CUtensorMap *tmK,
                                                 const CUtensorMap *tmV, int c) {
    using namespace sm100;
    AttendRowsBars &B = *reinterpret_cast<AttendRowsBars *>(smem + S::kOffBar);
    const int s = c % S::kStages;
    B.issued[s] = c / S::kStages + 1;
    const int tiles = min(S::kChunk / 128, (j.hi - j.lo - c * S::kChunk + 127) / 128);
    const bool last = j.hi - j.lo <= (c + 1) * S::kChunk;
    mbar_expect_tx(&B.full[s], 2 * kArTile * (uint32_t)tiles + (last ? g.debug_extra_tx : 0u));
#pragma unroll 1
    for (int t = 0; t < tiles; ++t) {
        const int key0 = j.lo + c * S::kChunk + t * 128;
        const int c1 = j.pos_t == 1 ? key0 : (j.pos_h == 1 ? j.h : j.b);
        const int c2 = j.pos_t == 2 ? key0 : (j.pos_h == 2 ? j.h : j.b);
        const int c3 = j.pos_t == 3 ? key0 : (j.pos_h == 3 ? j.h : j.b);
        uint8_t *dst = smem + kArOffStage + s * S::kStageBytes + t * kArTile;
        tma_load_4d(dst, tmK, &B.full[s], 0, c1, c2, c3);
        tma_load_4d(dst + S::kOffV, tmV, &B.full[s], 0, c1, c2, c3);
    }
}

// Thread kLoader: initialise the barriers and start the copies of the first `ahead` chunks.  They depend only on the
// unit and its length, not on the listed rows, so that a caller may run this early; the shared memory of the routine must
// be free.  In attend_rows_run the same thread (so that no block barrier is needed in between) starts the rest of the ring
// behind the loads of the query rows, which otherwise queue behind the copies of all CTAs (128 of them, K and V cold:
// 3.3 us instead of 2.1 us for the rows with three chunks ahead).
template <class S>
__device__ __forceinline__ void attend_rows_start(uint8_t *smem, const Geom &g, const AttendRowsJob &j,
                                                  const CUtensorMap *tmK, const CUtensorMap *tmV, int ahead) {
    using namespace sm100;
    AttendRowsBars &B = *reinterpret_cast<AttendRowsBars *>(smem + S::kOffBar);
    for (int s = 0; s < S::kStages; ++s) { mbar_init(&B.full[s], 1); B.left[s] = 0; B.issued[s] = 0; }
    B.abort_flag = 0;
    fence_barrier_init();
    const int n_chunks = (j.hi - j.lo + S::kChunk - 1) / S::kChunk;
#pragma unroll 1
    for (int c = 0; c < ahead && c < n_chunks; ++c) attend_rows_load<S>(smem, g, j, tmK, tmV, c);
}

// Not volatile, so that the compiler may place them; `epoch` (see ldmatrix_x4) ties them to the wait before them.
template <int OFF>
__device__ __forceinline__ void ar_ldmatrix(uint32_t addr, uint32_t epoch, uint32_t r[4]) {
    asm("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4 + %6]; // %5"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr), "r"(epoch), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ void ar_ldmatrix_t(uint32_t addr, uint32_t epoch, uint32_t r[4]) {
    asm("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4 + %6]; // %5"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr), "r"(epoch), "n"(OFF));
}
// (a, b) * scale + shift and a += b on both halves of a register pair
__device__ __forceinline__ float2 ar_fma2(float a, float b, float2 scale, float2 shift) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
        "fma.rn.f32x2 w, x, y, z;\n\tmov.b64 {%0, %1}, w;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a), "f"(b), "f"(scale.x), "f"(scale.y), "f"(shift.x), "f"(shift.y));
    return r;
}
__device__ __forceinline__ void ar_add2(float2 &a, float b0, float b1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a.x), "+f"(a.y) : "f"(b0), "f"(b1));
}
__device__ __forceinline__ uint32_t ar_pack(float a, float b) {
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&p);
}

// One warp: the key blocks grp, grp + groups, ... (32 keys each) for row tile `mt`.  m and l: reference and this lane's
// part of the weight sum of rows g and g + 8; o: C fragments of the 64 columns.
// The loop is kept short on purpose: unrolled over a chunk, or software pipelined (the scores of the next block ahead of the
// softmax of this one), the warps of a scheduler thrash its instruction cache: a third of the issue slots went to missing
// instructions, 7.5 and 10 us at T = 1024.  With 16 keys per trip instead of 32 the overhead of a trip weighs twice: 8.3 us.
template <class S>
__device__ __forceinline__ void attend_rows_warp(uint8_t *smem, const AttendRowsJob &j, const CUtensorMap *tmK,
                                                 const CUtensorMap *tmV, const Geom &g, int mt, int grp, int groups,
                                                 int n_warps, bool ones, float m[2], float l[2], float o[8][4]) {
    using namespace sm100;
    AttendRowsBars &B = *reinterpret_cast<AttendRowsBars *>(smem + S::kOffBar);
    const int lane = threadIdx.x & 31, l7 = lane & 7;
    const int n_keys = j.hi - j.lo, n_chunks = (n_keys + S::kChunk - 1) / S::kChunk, n_blocks = (n_keys + kArBlock - 1) / kArBlock;
    constexpr float kScaleLog2 = kScale * kLog2e;
    constexpr float kSlack = 8.f;                              // weights may grow to 2^8 before the reference moves
    uint32_t q[4][4], epoch;
    asm volatile("mov.u32 %0, 0;" : "=r"(epoch) :: "memory");
    {
        const int row = mt * 16 + l7 + 8 * ((lane >> 3) & 1);
        const uint32_t qa = smem_u32(smem + kArOffQ) + (uint32_t)row * 128u;
#pragma unroll
        for (int k = 0; k < 4; ++k) ldmatrix_x4(qa + ((uint32_t)((2 * k + (lane >> 4)) ^ l7) << 4), epoch, q[k][0], q[k][1], q[k][2], q[k][3]);
    }
    auto arrived = [&](int c) {                                // bounded wait, agreed on by the warp
        bool ok = *reinterpret_cast<volatile int *>(&B.abort_flag) == 0;
        if (ok) ok = mbar_wait(&B.full[c % S::kStages], (uint32_t)(c / S::kStages) & 1u, g.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok && lane == 0) { *reinterpret_cast<volatile int *>(&B.abort_flag) = 1; atomicOr(g.status, kStatusWaitExpired); }
        return ok;
    };
    // fragment addresses inside a block: K rows (l & 7) + 8 x, 16-byte chunks (l >> 3) and + 4 (the swizzled address with bit 6
    // flipped); V rows (l & 7) + 8 ((l >> 3) & 1) + 16 x, chunks 2 d + (l >> 4) (bits 5 and 6); a block starts at a
    // multiple of eight rows, so the swizzle depends on the lane alone
    const uint32_t base = smem_u32(smem + kArOffStage);
    const uint32_t k_lane = (uint32_t)l7 * 128u + ((uint32_t)((lane >> 3) ^ l7) << 4);
    const uint32_t v_lane = S::kOffV + (uint32_t)(l7 + 8 * ((lane >> 3) & 1)) * 128u + ((uint32_t)((lane >> 4) ^ l7) << 4);
    float2 l0 = make_float2(0.f, 0.f), l1 = l0;
    int c = -1, stage = -1, in_chunk = grp + S::kPerChunk;      // chunk, its stage, block inside it (normalised at the top)
    // Every warp passes every chunk in order, also one that holds no block of its group (one row tile: more groups than blocks per
    // chunk): a wait tells the two phases of a stage's barrier apart by parity only, so no warp may be two phases ahead of it, and a
    // stage is refilled when all warps have left it.
#pragma unroll 1
    for (int i = grp;; i += groups, in_chunk += groups) {
        while (in_chunk >= S::kPerChunk) {                      // on to the next chunk
            if (c >= 0 && c + S::kStages < n_chunks) {
#pragma unroll
                for (int x = 0; x < 8; ++x)                    // the fragments of the chunk have been read
                    asm volatile("" : "+f"(o[x][0]), "+f"(o[x][1]), "+f"(o[x][2]), "+f"(o[x][3]) :: "memory");
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    if (atomicAdd(&B.left[stage], 1) == n_warps - 1) { // the last warp to leave the stage refills it
                        B.left[stage] = 0;
                        __threadfence_block();
                        attend_rows_load<S>(smem, g, j, tmK, tmV, c + S::kStages);
                    }
                }
                __syncwarp();
            }
            in_chunk -= S::kPerChunk;
            if (++c >= n_chunks) break;
            stage = stage == S::kStages - 1 ? 0 : stage + 1;
            if (!arrived(c)) return;
        }
        if (i >= n_blocks) break;
        asm volatile("mov.u32 %0, %1;" : "=r"(epoch) : "r"(i) : "memory");
        const uint32_t at = base + (uint32_t)stage * S::kStageBytes + (uint32_t)in_chunk * (kArBlock * 128u);
        const int left = n_keys - i * kArBlock;                // keys from the block's first on
        float s[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[x][e] = 0.f;
        if (!ones) {
            const uint32_t k0 = at + k_lane, k1 = k0 ^ 64u;
            uint32_t k[4][8];
            ar_ldmatrix<0>(k0, epoch, k[0]); ar_ldmatrix<0>(k1, epoch, k[0] + 4);
            ar_ldmatrix<1024>(k0, epoch, k[1]); ar_ldmatrix<1024>(k1, epoch, k[1] + 4);
            ar_ldmatrix<2048>(k0, epoch, k[2]); ar_ldmatrix<2048>(k1, epoch, k[2] + 4);
            ar_ldmatrix<3072>(k0, epoch, k[3]); ar_ldmatrix<3072>(k1, epoch, k[3] + 4);
#pragma unroll
            for (int x = 0; x < 4; ++x) mma_bf16_16816_first(s[x], q[0][0], q[0][1], q[0][2], q[0][3], k[x][0], k[x][1]);
#pragma unroll
            for (int t = 1; t < 4; ++t)
#pragma unroll
                for (int x = 0; x < 4; ++x) mma_bf16_16816(s[x], q[t][0], q[t][1], q[t][2], q[t][3], k[x][2 * t], k[x][2 * t + 1]);
        }
        if (left < kArBlock) {
            // the end of the sequence: weight exp2(-inf) = 0; the rows of V behind it, which may hold anything (even NaN),
            // become zero, so that 0 * x stays 0 (the other row tiles' warps write the same zeros)
            const int k0 = 2 * (lane & 3);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (k0 + 8 * x >= left) { s[x][0] = -INFINITY; s[x][2] = -INFINITY; }
                if (k0 + 8 * x + 1 >= left) { s[x][1] = -INFINITY; s[x][3] = -INFINITY; }
            }
#pragma unroll 1
            for (int e = left * 8 + lane; e < kArBlock * 8; e += 32)
                asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(at + S::kOffV + (uint32_t)e * 16u), "r"(0) : "memory");
            __syncwarp();
            asm volatile("mov.u32 %0, %1;" : "=r"(epoch) : "r"(i) : "memory");
        }
        float t0 = fmaxf(s[0][0], s[0][1]), t1 = fmaxf(s[0][2], s[0][3]);
#pragma unroll
        for (int x = 1; x < 4; ++x) { t0 = fmaxf(t0, fmaxf(s[x][0], s[x][1])); t1 = fmaxf(t1, fmaxf(s[x][2], s[x][3])); }
        t0 *= kScaleLog2; t1 *= kScaleLog2;
        if (__any_sync(0xffffffffu, t0 > m[0] + kSlack || t1 > m[1] + kSlack)) {       // always so in the first block (m = -inf)
            float n0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 1)), n1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 1));
            n0 = fmaxf(n0, __shfl_xor_sync(0xffffffffu, n0, 2)); n1 = fmaxf(n1, __shfl_xor_sync(0xffffffffu, n1, 2));
            n0 = fmaxf(n0, m[0]); n1 = fmaxf(n1, m[1]);
            const float a0 = fast_exp2(m[0] - n0), a1 = fast_exp2(m[1] - n1);          // 0 the first time
            l0.x *= a0; l0.y *= a0; l1.x *= a1; l1.y *= a1; m[0] = n0; m[1] = n1;
#pragma unroll
            for (int x = 0; x < 8; ++x) { o[x][0] *= a0; o[x][1] *= a0; o[x][2] *= a1; o[x][3] *= a1; }
        }
        uint32_t p[4][2];                                      // of eight keys: rows g and g + 8
        const float2 sc = make_float2(kScaleLog2, kScaleLog2), m0 = make_float2(-m[0], -m[0]), m1 = make_float2(-m[1], -m[1]);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            float2 w0 = ar_fma2(s[x][0], s[x][1], sc, m0), w1 = ar_fma2(s[x][2], s[x][3], sc, m1);
            w0.x = fast_exp2(w0.x); w0.y = fast_exp2(w0.y); w1.x = fast_exp2(w1.x); w1.y = fast_exp2(w1.y);
            ar_add2(l0, w0.x, w0.y); ar_add2(l1, w1.x, w1.y);
            p[x][0] = ar_pack(w0.x, w0.y); p[x][1] = ar_pack(w1.x, w1.y);
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const uint32_t va = (at + v_lane) ^ (uint32_t)(d << 5);
            uint32_t v[4], w[4];
            ar_ldmatrix_t<0>(va, epoch, v);
            ar_ldmatrix_t<2048>(va, epoch, w);
            mma_bf16_16816(o[2 * d], p[0][0], p[0][1], p[1][0], p[1][1], v[0], v[1]);
            mma_bf16_16816(o[2 * d + 1], p[0][0], p[0][1], p[1][0], p[1][1], v[2], v[3]);
            mma_bf16_16816(o[2 * d], p[2][0], p[2][1], p[3][0], p[3][1], w[0], w[1]);
            mma_bf16_16816(o[2 * d + 1], p[2][0], p[2][1], p[3][0], p[3][1], w[2], w[3]);
        }
    }
    l[0] = l0.x + l0.y; l[1] = l1.x + l1.y;
}

// All threads of the CTA (contains __syncthreads); attend_rows_start must have been run with the same
// `ahead`.  On return thread t holds, of
// rows t / 8 + x kThreads / 8, the softmax state over [lo, hi): m (scaled log2 units), l, and the unnormalised columns 8 (t % 8) .. + 7.
// Returns false if a wait ran out (status bit set).
template <class S>
__device__ __forceinline__ bool attend_rows_run(uint8_t *smem, const Geom &g, const AttendRowsJob &j,
                                                const __nv_bfloat16 *__restrict__ Q, const CUtensorMap *tmK,
                                                const CUtensorMap *tmV, int ahead, float (&m_out)[S::kRows],
                                                float (&l_out)[S::kRows], float (&acc)[S::kRows][8]) {
    using namespace sm100;
    AttendRowsBars &B = *reinterpret_cast<AttendRowsBars *>(smem + S::kOffBar);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {   // the listed rows of Q, 16-byte pieces; unused rows are zero
        uint4 v[S::kRows];
#pragma unroll
        for (int x = 0; x < S::kRows; ++x) {
            const int r = (tid + x * S::kThreads) >> 3, c = tid & 7;
            int i = -1;
            if (r < j.n_rows) i = j.rows ? j.rows[r] : r;
            v[x] = make_uint4(0u, 0u, 0u, 0u);
            if (i >= 0 && i < j.L)
                v[x] = __ldg(reinterpret_cast<const uint4 *>(Q + unit_off(g.qs, j.b, j.h) + (long long)i * g.qs[2]) + c);
        }
        if (tid == S::kLoader) {
            const int n_chunks = (j.hi - j.lo + S::kChunk - 1) / S::kChunk;
#pragma unroll 1
            for (int x = ahead; x < S::kStages && x < n_chunks; ++x) attend_rows_load<S>(smem, g, j, tmK, tmV, x);
        }
#pragma unroll
        for (int x = 0; x < S::kRows; ++x) {
            const int r = (tid + x * S::kThreads) >> 3, c = tid & 7;
            *reinterpret_cast<uint4 *>(smem + kArOffQ + r * 128 + ((c ^ (r & 7)) << 4)) = v[x];
        }
    }
    __syncthreads();
    phase_stamp(g, 6);
    const int used = max(j.n_rows, j.sum_row + 1), tiles = (used + 15) / 16;
    const int groups = (S::kThreads / 32) / max(tiles, 1);     // of 16 warps: 16, 8, 5, 4
    const int mt = warp / groups, grp = warp % groups;
    const bool ones = j.sum_row >= 0 && mt * 16 >= j.n_rows;   // a tile with no query but the all-ones row
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, o[8][4];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[x][e] = 0.f;
    if (mt < tiles) {
        attend_rows_warp<S>(smem, j, tmK, tmV, g, mt, grp, groups, groups * tiles, ones, m, l, o);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
    }
    __syncthreads();
    phase_stamp(g, 7);
    const bool ok = *reinterpret_cast<volatile int *>(&B.abort_flag) == 0;
    if (!ok) {
        // copies that were issued but never consumed: give them a bounded chance to land
        if (tid == 0)
            for (int s = 0; s < S::kStages; ++s)
                if (B.issued[s] > 0) {
                    mbar_wait(&B.full[s], (uint32_t)(B.issued[s] - 1) & 1u, g.wait_ns);
                }
        __syncthreads();
#pragma unroll
        for (int y = 0; y < S::kRows; ++y) {
            m_out[y] = -INFINITY; l_out[y] = 0.f;
#pragma unroll
            for (int x = 0; x < 8; ++x) acc[y][x] = 0.f;
        }
        return false;
    }
    // merge: state of (group, row) at [group][row][kArPitch] in the stages' memory, which nobody reads any more
    float *buf = reinterpret_cast<float *>(smem + kArOffStage);
    const int rows = tiles * 16;
    if (mt < tiles) {
        float *lo = buf + (grp * rows + mt * 16 + (lane >> 2)) * kArPitch, *hi = lo + 8 * kArPitch;
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            *reinterpret_cast<float2 *>(lo + 8 * x + 2 * (lane & 3)) = make_float2(o[x][0], o[x][1]);
            *reinterpret_cast<float2 *>(hi + 8 * x + 2 * (lane & 3)) = make_float2(o[x][2], o[x][3]);
        }
        if ((lane & 3) == 0) { lo[64] = m[0]; lo[65] = l[0]; hi[64] = m[1]; hi[65] = l[1]; }
    }
    __syncthreads();
    const int c8 = tid & 7;
#pragma unroll
    for (int y = 0; y < S::kRows; ++y) {
        const int r = (tid + y * S::kThreads) >> 3;
        float mw = -INFINITY, lw = 0.f;
#pragma unroll
        for (int x = 0; x < 8; ++x) acc[y][x] = 0.f;
        if (r < rows) {
            for (int x = 0; x < groups; ++x) mw = fmaxf(mw, buf[(x * rows + r) * kArPitch + 64]);
#pragma unroll 4
            for (int x = 0; x < groups; ++x) {
                const float *src = buf + (x * rows + r) * kArPitch;
                const float f = src[65] > 0.f ? fast_exp2(src[64] - mw) : 0.f;
                const float4 u = *reinterpret_cast<const float4 *>(src + 8 * c8), v = *reinterpret_cast<const float4 *>(src + 8 * c8 + 4);
                lw += src[65] * f;
                acc[y][0] = fmaf(u.x, f, acc[y][0]); acc[y][1] = fmaf(u.y, f, acc[y][1]); acc[y][2] = fmaf(u.z, f, acc[y][2]); acc[y][3] = fmaf(u.w, f, acc[y][3]);
                acc[y][4] = fmaf(v.x, f, acc[y][4]); acc[y][5] = fmaf(v.y, f, acc[y][5]); acc[y][6] = fmaf(v.z, f, acc[y][6]); acc[y][7] = fmaf(v.w, f, acc[y][7]);
            }
        }
        m_out[y] = mw; l_out[y] = lw;
    }
    return true;
}

}  // namespace psattn
