// Float32 steps with hydrodynamic interaction (Eqs. 1-3) whose Cholesky
// factorisation of the Rotne-Prager-Yamakawa tensor W runs its trailing
// updates on the tensor cores.
//
// One CTA of 160 threads integrates one slot of a chain of N <= 50 beads
// (n = 3N <= 150 rows of W). The last m = n - t0 <= 126 rows and columns of W
// (t0 = 3 max(0, N - 42), a bead boundary) form the trailing block T, held in
// tensor memory (TMEM): thread i of warps 0-3 owns row i of T, TMEM lane i.
// The first t0 <= 24 rows (the head) belong to the lanes of warp 4. Per step:
//   - bead forces and normals (as the CUDA-core kernel), and W's blocks (Eqs.
//     2-3), one bead pair a thread, into a shared copy of T;
//   - every thread takes its own row of the copy, the mobility-weighted force
//     u = (W F)_row on the way, and stores it to its TMEM lane; the head
//     columns follow through the same place into registers;
//   - head: warp 4 factors the head block (one row a lane, four columns at a
//     time, their entries through shared memory); the
//     T rows solve their head columns against it (X L^T = W_T,head) and
//     T <- T - X X^T on the tensor cores;
//   - panels of 32 columns of T: warp p factors the diagonal block of
//     panel p (its 32 rows), the rows below solve against it, and the
//     tensor cores subtract the panel's outer product from the rest of T;
//     that update is issued as the next panel's 32 columns first and the
//     remaining columns after, so the next panel's factor starts as soon as
//     its own columns are done;
//   - the correlated noise w = L xi accumulates row by row as the factor's
//     entries appear; then the update and the centre-of-mass shift.
// The MMAs are kind::tf32 with float32 accumulators in TMEM, every product
// of float32 values split as hi hi + hi lo + lo hi (tf32 high parts and
// remainders), which keeps the float32 accuracy of the factor. Completion is
// tracked by two mbarriers whose waits give up after a bounded number of
// polls: the CTA then records BD_DEV_ERR_TC_WAIT, stops integrating, waits
// (bounded) for its MMAs and frees its TMEM.
#pragma once

#include "bd_hi.cuh"
#include "bd_tc.cuh"

namespace bdra {

constexpr int kTCThreads = 160;          // four row warps (TMEM lanes 0-127) + the head warp
constexpr int kTCMaxBeads = kHISmallBeads;
constexpr int kTCHeadBeads = 8;          // head of at most 24 rows
constexpr uint32_t kTCCols = 128;        // TMEM columns of a CTA
constexpr int kTCBlocksPerSM = 3;        // CTAs an SM holds (128 registers a thread; TMEM would allow 4)
static_assert(kTCBlocksPerSM * kTCCols <= 512, "TMEM columns of the resident CTAs");
constexpr uint32_t kTCPolls = 1u << 20;  // polls of a completion barrier before giving up
static_assert(3 * (kTCMaxBeads - 42) <= 3 * kTCHeadBeads, "head of the largest chain");

constexpr int kTCRows = 126;             // rows of the trailing block at most (42 beads)
constexpr int kTCStride = 132;           // row strides of the tensor's shared copies: 16-byte rows whose
constexpr int kTCHeadStride = 28;        // vector loads, one row a lane, meet every bank once

constexpr int kTCNB = 4;                 // columns the diagonal factor takes at a time (8: spills, 8% slower)

struct HITCShared {
    // W's trailing block while it is assembled, then its head columns (every
    // row of the chain), then the MMA operands
    union alignas(128) {
        float w[kTCRows * kTCStride];
        float wh[3 * kTCMaxBeads * kTCHeadStride];
        struct {
            alignas(128) float op_hi[128 * 32];  // the panel's factor rows (tf32 high parts), MMA operand layout
            alignas(128) float op_lo[128 * 32];  // their remainders
        };
    };
    alignas(16) float lt[32][32];        // factor of the current diagonal block, transposed: lt[k][j] = L[j][k]
    alignas(16) float col[2][kTCNB][32]; // columns of the block being factored (two sets in flight)
    alignas(16) float dinv[32];          // reciprocals of its diagonal
    alignas(16) float pos[4 * kHINTSmall];   // bead positions [3N] (COM frame)
    alignas(16) float frc[4 * kHINTSmall];   // bead forces [3N]
    alignas(16) float xi[4 * kHINTSmall];    // bead normals [3N]
    float com[3];
    // bead pairs bi >= bj as (bi << 8) | bj: those of the trailing block in row
    // order, then those with a head bead
    uint16_t pr[kTCMaxBeads * (kTCMaxBeads + 1) / 2];
    uint32_t taddr;                      // TMEM address of the CTA's columns
    alignas(8) uint64_t bar_next;        // MMAs of the next panel's columns done
    alignas(8) uint64_t bar_rest;        // MMAs of the columns after them done
};

// Per-thread bookkeeping of the CTA's tensor-memory state. Only thread 0
// (which issues the MMAs) waits on the completion barriers and tracks their
// phases; a CTA barrier then passes the completion on to the other threads.
struct TCState {
    uint32_t taddr;      // this warp's lanes (row warps), first column
    uint32_t ph_next, ph_rest;
    bool pend_next, pend_rest;
    bool bad;            // a wait gave up
    bool stall;          // BD_FLAG_TEST_TC_STALL: no MMA and no completion is issued
    int t0, m, hb, P;    // head rows, T rows, head beads, panels

    __device__ __forceinline__ void setup(int N)
    {
        const int n = 3 * N;
        hb = N > 42 ? N - 42 : 0;
        t0 = 3 * hb;
        m = n - t0;
        P = (m + 31) >> 5;
        ph_next = ph_rest = 0;
        pend_next = pend_rest = false;
        bad = false;
    }
    __device__ __forceinline__ void wait_next(HITCShared& sm)
    {
        if (threadIdx.x != 0 || !pend_next) return;
        if (!tc::mbar_wait(&sm.bar_next, ph_next, kTCPolls)) bad = true;
        ph_next ^= 1u;
        pend_next = false;
    }
    __device__ __forceinline__ void wait_rest(HITCShared& sm)
    {
        if (threadIdx.x != 0 || !pend_rest) return;
        if (!tc::mbar_wait(&sm.bar_rest, ph_rest, kTCPolls)) bad = true;
        ph_rest ^= 1u;
        pend_rest = false;
    }
};

// The 3 x 3 blocks of W (Eqs. 2-3) of the bead pairs q0 <= q < q1 of sm.pr
// into a shared copy of rows of `stride` floats, both triangles: the block of
// a pair is c_d d d^T + c_i I (d = r_bj - r_bi, c_d > 0 in both branches of
// Eq. 3), taken as e e^T + c_i I with e = sqrt(c_d) d, so that transposed
// entries are equal bitwise; the diagonal blocks are the identity. Row r of W
// is row r - r0 of the copy, columns start at column c0 of W and end before c1
// (head columns: only one of a block's two places may lie inside).
//
// A pair a thread and whole rows back: building its own row bead by bead took
// each thread 30 instructions a bead (coefficient load, selects, three broadcast
// loads), 26% of a step; the copy costs a thread six pairs of 18 stores and a
// row of 32 vector loads. It lies where the MMA operands come later.
__device__ __forceinline__ void tc_blocks(HITCShared& sm, float* dst, int stride, int r0, int c0, int c1, int q0, int q1,
                                          float a)
{
#pragma unroll 1
    for (int q = q0 + (int)threadIdx.x; q < q1; q += kTCThreads) {
        const int bi = sm.pr[q] >> 8, bj = sm.pr[q] & 0xFF;
        float e[3], ci;
        if (bi == bj) {
            e[0] = e[1] = e[2] = 0.0f;
            ci = 1.0f;
        } else {
            const float dx = sm.pos[3 * bj] - sm.pos[3 * bi];
            const float dy = sm.pos[3 * bj + 1] - sm.pos[3 * bi + 1];
            const float dz = sm.pos[3 * bj + 2] - sm.pos[3 * bi + 2];
            float cd;
            rpy_coef<float, true>(dx, dy, dz, a, ci, cd);
            const float sc = sqrt_approx(cd);
            e[0] = sc * dx; e[1] = sc * dy; e[2] = sc * dz;
        }
        const bool lower = 3 * bj >= c0 && 3 * bj < c1, upper = 3 * bi >= c0 && 3 * bi < c1;
        float* lo = dst + (3 * bi - r0) * stride + 3 * bj - c0;      // rows of bi, columns of bj
        float* up = dst + (3 * bj - r0) * stride + 3 * bi - c0;
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                const float w = __fmaf_rn(e[x], e[y], x == y ? ci : 0.0f);
                if (lower) lo[x * stride + y] = w;
                if (upper) up[y * stride + x] = w;
            }
    }
}

// The pair table (once per kernel): pairs of trailing beads (bj >= hb), then
// those with a head bead.
__device__ __forceinline__ void tc_pairs_init(HITCShared& sm, int N, int hb)
{
    const int m = N - hb, trailing = m * (m + 1) / 2;
    for (int q = threadIdx.x; q < N * (N + 1) / 2; q += blockDim.x) {
        int bi, bj;
        if (q < trailing) {
            hi_untri(q, bi, bj);
            bi += hb; bj += hb;
        } else {                   // bj < hb: bead bi = 0, 1, .. with min(bi + 1, hb) partners each
            const int h = q - trailing, tri = hb * (hb + 1) / 2;
            if (h < tri) {
                hi_untri(h, bi, bj);
            } else {
                bi = hb + (h - tri) / hb;
                bj = (h - tri) % hb;
            }
        }
        sm.pr[q] = (uint16_t)((bi << 8) | bj);
    }
}

// Lower Cholesky factor of a K x K block held one row a lane (A[j], j < K;
// rows beyond the block are identity rows), NB columns at a time (K a multiple
// of NB, NB of 4). The columns are a serial chain and one warp works on it, so
// its latency is all that counts: a column by itself is a reciprocal root on
// its owner, a shuffle, and a pass of the column through shared memory before
// the next root's entry is right (140 cycles). The NB x NB diagonal block's
// lower entries are shuffled to every lane instead, each lane factors it by
// itself (NB roots, no exchange between them), solves its own NB entries
// against it, and the columns pass through shared memory together for the
// update of the later ones, the next NB first: the rest of it fills the next
// block's waits. Every entry takes the same operations in the same order as
// column by column. Returns 1 / L[lane][lane].
template <int K>
__device__ __forceinline__ float tc_warp_chol(float (&A)[32], int lane, float (*col)[kTCNB][32])
{
    constexpr int NB = kTCNB;
    float own_inv = 1.0f;
    float x[NB];
    // columns j4 .. j4 + 3 of the update by the NB columns in buf
    auto update = [&](const float (&buf)[NB][32], int j4) {
#pragma unroll
        for (int c = 0; c < NB; ++c) {
            const float4 l = *reinterpret_cast<const float4*>(&buf[c][j4]);
            A[j4 + 0] = __fmaf_rn(-x[c], l.x, A[j4 + 0]);
            A[j4 + 1] = __fmaf_rn(-x[c], l.y, A[j4 + 1]);
            A[j4 + 2] = __fmaf_rn(-x[c], l.z, A[j4 + 2]);
            A[j4 + 3] = __fmaf_rn(-x[c], l.w, A[j4 + 3]);
        }
    };
#pragma unroll
    for (int k = 0; k < K; k += NB) {
        float d[NB][NB], il[NB];
#pragma unroll
        for (int r = 0; r < NB; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) d[r][c] = __shfl_sync(0xffffffffu, A[k + c], k + r);
        if (k > 0) {
#pragma unroll
            for (int j4 = k + NB; j4 < K; j4 += 4) update(col[((k / NB) + 1) & 1], j4);
        }
#pragma unroll
        for (int c = 0; c < NB; ++c) {
            il[c] = Rsqrt<float, true>::rsqrt(d[c][c]);
#pragma unroll
            for (int r = c + 1; r < NB; ++r) d[r][c] = __fmul_rn(d[r][c], il[c]);
#pragma unroll
            for (int c2 = c + 1; c2 < NB; ++c2)
#pragma unroll
                for (int r = c2; r < NB; ++r) d[r][c2] = __fmaf_rn(-d[r][c], d[c2][c], d[r][c2]);
        }
        // the lane's entries of the columns: below its diagonal the solve, on it
        // the root, above it what was there (never used)
#pragma unroll
        for (int c = 0; c < NB; ++c) {
            float v = A[k + c];
#pragma unroll
            for (int c2 = 0; c2 < c; ++c2) v = __fmaf_rn(-x[c2], d[c][c2], v);
            x[c] = lane >= k + c ? __fmul_rn(v, il[c]) : 0.0f;
            if (lane == k + c) own_inv = il[c];
            if (lane >= k + c) A[k + c] = x[c];
        }
        if (k + NB < K) {
            float (&buf)[NB][32] = col[(k / NB) & 1];
#pragma unroll
            for (int c = 0; c < NB; ++c) buf[c][lane] = x[c];
            __syncwarp();
#pragma unroll
            for (int j4 = k + NB; j4 < k + 2 * NB; j4 += 4) update(buf, j4);
        }
    }
    return own_inv;
}

// A <- A L^{-T} (forward substitution over K columns, four at a time) with the
// factor in sm.lt / sm.dinv; columns whose factor rows are identity rows pass
// through.
template <int K>
__device__ __forceinline__ void tc_row_solve(float (&A)[32], const HITCShared& sm)
{
#pragma unroll
    for (int k = 0; k < K; k += 4) {
        const float4 iv = *reinterpret_cast<const float4*>(&sm.dinv[k]);
        const float4 l0 = *reinterpret_cast<const float4*>(&sm.lt[k][k]);
        const float4 l1 = *reinterpret_cast<const float4*>(&sm.lt[k + 1][k]);
        const float4 l2 = *reinterpret_cast<const float4*>(&sm.lt[k + 2][k]);
        A[k] = __fmul_rn(A[k], iv.x);
        A[k + 1] = __fmul_rn(__fmaf_rn(-A[k], l0.y, A[k + 1]), iv.y);
        A[k + 2] = __fmul_rn(__fmaf_rn(-A[k + 1], l1.z, __fmaf_rn(-A[k], l0.z, A[k + 2])), iv.z);
        A[k + 3] = __fmul_rn(__fmaf_rn(-A[k + 2], l2.w, __fmaf_rn(-A[k + 1], l1.w, __fmaf_rn(-A[k], l0.w, A[k + 3]))), iv.w);
#pragma unroll
        for (int j4 = k + 4; j4 < K; j4 += 4)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 l = *reinterpret_cast<const float4*>(&sm.lt[k + c][j4]);
                A[j4 + 0] = __fmaf_rn(-A[k + c], l.x, A[j4 + 0]);
                A[j4 + 1] = __fmaf_rn(-A[k + c], l.y, A[j4 + 1]);
                A[j4 + 2] = __fmaf_rn(-A[k + c], l.z, A[j4 + 2]);
                A[j4 + 3] = __fmaf_rn(-A[k + c], l.w, A[j4 + 3]);
            }
    }
}

// Row `row` of the MMA operand (tf32 split) from A[0 .. 4 nc).
template <int NC>
__device__ __forceinline__ void tc_put_operand(HITCShared& sm, int row, const float (&A)[32], bool zero)
{
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        float h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (zero) h[e] = l[e] = 0.0f;
            else tc::split_tf32(A[4 * c + e], h[e], l[e]);
        }
        const int o = tc::op_index(row, 4 * c, 8);
        *reinterpret_cast<float4*>(&sm.op_hi[o]) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4*>(&sm.op_lo[o]) = make_float4(l[0], l[1], l[2], l[3]);
    }
}

// T[:, c0 .. c0 + N) -= X X[c0 .. c0 + N)^T over ks K steps of 8, X
// the operand rows (three tf32 products per step). The descriptors of all
// steps are the first one's plus 256 bytes a step (address field in 16 bytes).
__device__ __forceinline__ void tc_issue_update(HITCShared& sm, uint32_t tbase, int c0, int N, int ks)
{
    const uint32_t id = tc::idesc_tf32(128, N, true);
    const uint32_t hi = tc::smem_u32(sm.op_hi), lo = tc::smem_u32(sm.op_lo);
    const uint32_t boff = (uint32_t)(c0 >> 3) * 1024u, d = tbase + (uint32_t)c0;
    const uint64_t ah = tc::smem_desc(hi, 128, 1024), al = tc::smem_desc(lo, 128, 1024);
    const uint64_t bh = tc::smem_desc(hi + boff, 128, 1024), bl = tc::smem_desc(lo + boff, 128, 1024);
#pragma unroll 1                             // (unrolled: 1.5% slower)
    for (int s = 0; s < ks; ++s) {
        tc::mma_tf32(d, ah + 16 * s, bh + 16 * s, id, true);
        tc::mma_tf32(d, ah + 16 * s, bl + 16 * s, id, true);
        tc::mma_tf32(d, al + 16 * s, bh + 16 * s, id, true);
    }
}

// The two-part update after a panel (or the head): thread 0 issues the next
// panel's columns [c1, c1 + 32) and its completion (bar_next), thread
// kTCSecond the rest up to the padded width of T (bar_rest): one thread
// needs 2000 cycles to issue all 24 MMAs, longer than they run (800). With `stall` (a
// failure test) nothing is issued, so the waits give up.
constexpr int kTCSecond = 128;
__device__ __forceinline__ void tc_issue_two(HITCShared& sm, uint32_t tbase, int c1, int m, int ks, bool stall)
{
    if (stall) return;
    if (threadIdx.x == 0) {
        tc::fence_after_sync();
        tc_issue_update(sm, tbase, c1, 32, ks);
        tc::mma_commit(&sm.bar_next);
    } else if (threadIdx.x == kTCSecond) {
        tc::fence_after_sync();
        const int width = (m + 15) & ~15;
        if (c1 + 32 < width) tc_issue_update(sm, tbase, c1 + 32, width - c1 - 32, ks);
        tc::mma_commit(&sm.bar_rest);
    }
}

__device__ __forceinline__ void tc_sync()
{
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// One step t -> t + 1 of the CTA's slot (float32). Returns the thread's
// FENE floor count; ts.bad is set (on every thread) if a wait gave up.
__device__ __forceinline__ int hi_tc_step(HITCShared& sm, TCState& ts, const ChainDev& ch,
                                          const StepConst<float, true>& k, const LJConst<float>& kl,
                                          const StepParams& p, int N,
                                          uint32_t slot_key, uint32_t chain, uint32_t step, bool harmonic, bool lj)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t0 = ts.t0, m = ts.m, hb = ts.hb, P = ts.P;
    const int floored = hi_forces<float, true>(sm, N, k, kl, harmonic, lj);
    // the normals on the last threads: the force pass's second round (beads past
    // the 40th) keeps the first warps
    if (const int b = tid - (kTCThreads - N); b >= 0) {
        float z0, z1, z2;
        bead_noise<float, true>((uint32_t)b, slot_key, step, chain, p, z0, z1, z2);
        sm.xi[3 * b] = z0;
        sm.xi[3 * b + 1] = z1;
        sm.xi[3 * b + 2] = z2;
    }
    const int trailing = (N - hb) * (N - hb + 1) / 2;       // pairs of trailing beads
    tc_blocks(sm, sm.w, kTCStride, t0, t0, 3 * N, 0, trailing, (float)ch.hi_a);
    __syncthreads();

    // rows of W: T rows (warps 0-3) into TMEM, then their head columns into
    // registers; head rows (warp 4): the head block into registers, the rest
    // of the row for u only
    const bool head = warp == 4;
    const int row = head ? lane : t0 + tid;
    const bool valid = head ? lane < t0 : tid < m;
    float A[32];
    float w = 0.0f;
    float u[3] = {0.0f, 0.0f, 0.0f};           // (W F)_row over the columns of each component, bead by bead
    if (!head) {
        const float* src = sm.w + (valid ? tid : 0) * kTCStride;
#pragma unroll
        for (int g = 0; g < 16; ++g) {         // TMEM columns [8 g, 8 g + 8)
            float V[8];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 v = *reinterpret_cast<const float4*>(src + 8 * g + 4 * q);
                V[4 * q] = v.x; V[4 * q + 1] = v.y; V[4 * q + 2] = v.z; V[4 * q + 3] = v.w;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int c = 8 * g + e;
                if (!(valid && c < m)) V[e] = 0.0f;      // past the block the copy holds anything
                if (c < kTCRows) u[c % 3] = __fmaf_rn(V[e], sm.frc[t0 + c], u[c % 3]);
            }
            tc::tmem_st8(ts.taddr + 8 * g, V);
        }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) A[j] = 0.0f;
    if (t0 > 0) {                              // (t0 is the CTA's)
        __syncthreads();                       // the trailing block is read: its place takes the head columns
        tc_blocks(sm, sm.wh, kTCHeadStride, 0, 0, t0, trailing, N * (N + 1) / 2, (float)ch.hi_a);
        __syncthreads();
        if (head && valid) {
#pragma unroll 7
            for (int c = t0; c < 3 * N; c += 3) {          // the row's trailing columns, by symmetry
                u[0] = __fmaf_rn(sm.wh[c * kTCHeadStride + lane], sm.frc[c], u[0]);
                u[1] = __fmaf_rn(sm.wh[(c + 1) * kTCHeadStride + lane], sm.frc[c + 1], u[1]);
                u[2] = __fmaf_rn(sm.wh[(c + 2) * kTCHeadStride + lane], sm.frc[c + 2], u[2]);
            }
        }
        const float* src = sm.wh + (valid ? row : 0) * kTCHeadStride;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(src + 4 * q);
            A[4 * q] = v.x; A[4 * q + 1] = v.y; A[4 * q + 2] = v.z; A[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int c = 0; c < 3 * kTCHeadBeads; ++c) {
            if (!(valid && c < t0)) A[c] = 0.0f;
            u[c % 3] = __fmaf_rn(A[c], sm.frc[c], u[c % 3]);
        }
    }
    const float uf = __fadd_rn(__fadd_rn(u[0], u[1]), u[2]);
    if (head && !valid) {        // identity rows below the head block
#pragma unroll
        for (int j = 0; j < 32; ++j) A[j] = j == lane ? 1.0f : 0.0f;
    }
    if (!head) tc::tmem_wait_st();
    tc_sync();

    // head: factor (warp 4), solve of the T rows, T -= X X^T
    if (t0 > 0) {
        if (head) {
            const float il = tc_warp_chol<3 * kTCHeadBeads>(A, lane, sm.col);
#pragma unroll
            for (int j = 0; j < 3 * kTCHeadBeads; ++j) sm.lt[j][lane] = A[j];
            sm.dinv[lane] = il;
        }
        __syncthreads();
        if (!head) {
            tc_row_solve<3 * kTCHeadBeads>(A, sm);
            tc_put_operand<2 * kTCHeadBeads * 3 / 8>(sm, tid, A, !valid);
        }
        tc::fence_async_smem();
        __syncthreads();
        tc_issue_two(sm, ts.taddr & 0xFFFFu, 0, m, (t0 + 7) >> 3, ts.stall);
        ts.pend_next = ts.pend_rest = true;
        // w = L xi, here and in the panels behind the barrier that others wait at
        // (rows past T are zero rows in the head columns)
#pragma unroll
        for (int j = 0; j < 3 * kTCHeadBeads; ++j)
            if (!head || (valid && j <= lane)) w = __fmaf_rn(A[j], sm.xi[j], w);
    }

    // panels of T
#pragma unroll 1
    for (int pn = 0; pn < P; ++pn) {
        const int c0 = 32 * pn;
        ts.wait_next(sm);
        tc_sync();                 // the next panel's columns are in TMEM
        if (!head) {
            if (warp >= pn) {
                tc::tmem_ld32(ts.taddr + (uint32_t)c0, A);
                if (!valid) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) A[j] = c0 + j == tid ? 1.0f : 0.0f;
                }
            }
            if (warp == pn) {
                const float il = tc_warp_chol<32>(A, lane, sm.col);
#pragma unroll
                for (int j = 0; j < 32; ++j) sm.lt[j][lane] = A[j];
                sm.dinv[lane] = il;
            }
        }
        ts.wait_rest(sm);          // the previous update no longer reads the operand
        tc_sync();
        if (!head && warp > pn) tc_row_solve<32>(A, sm);
        if (pn + 1 < P) {
            if (!head && warp > pn) tc_put_operand<8>(sm, tid, A, !valid);
            tc::fence_async_smem();
            __syncthreads();
            tc_issue_two(sm, ts.taddr & 0xFFFFu, c0 + 32, m, 4, ts.stall);
            ts.pend_next = ts.pend_rest = true;
        } else {
            __syncthreads();       // every read of sm.lt done before the next step writes it
        }
        if (!head && warp >= pn && valid)
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (warp > pn || j <= lane) w = __fmaf_rn(A[j], sm.xi[t0 + c0 + j], w);
    }
    ts.wait_next(sm);
    ts.wait_rest(sm);
    tc::fence_before_sync();
    ts.bad = __syncthreads_or(ts.bad) != 0;    // every MMA of the step is done
    tc::fence_after_sync();

    // update and centre-of-mass shift
    float nv = 0.0f;
    if (valid) {
        const int xx = row % 3, b3 = row - xx;
        const float r = sm.pos[row];
        const float fl = xx == 0 ? fmaf(k.axz, sm.pos[b3 + 2], fmaf(k.axx, r, r))
                                 : (xx == 1 ? fmaf(k.ayy, r, r) : fmaf(k.azz, r, r));
        nv = fmaf(k.cn, w, fmaf(k.cd, uf, fl));
    }
    __syncthreads();
    if (valid) sm.pos[row] = nv;
    __syncthreads();
    if (tid < 32) {
        float s[3] = {0.0f, 0.0f, 0.0f};
        for (int b = tid; b < N; b += 32)
#pragma unroll
            for (int c = 0; c < 3; ++c) s[c] += sm.pos[3 * b + c];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
        }
        if (tid == 0)
#pragma unroll
            for (int c = 0; c < 3; ++c) sm.com[c] = s[c] / (float)N;
    }
    __syncthreads();
    if (tid < 3 * N) sm.pos[tid] -= sm.com[tid % 3];
    __syncthreads();
    return floored;
}

// Set-up of a CTA: barriers and TMEM columns (warp 0); every thread's state.
__device__ __forceinline__ void hi_tc_begin(HITCShared& sm, TCState& ts, int N)
{
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        tc::mbar_init(&sm.bar_next, 1);
        tc::mbar_init(&sm.bar_rest, 1);
    }
    tc_pairs_init(sm, N, N > 42 ? N - 42 : 0);
    if (warp == 0) {
        tc::tmem_alloc(&sm.taddr, kTCCols);
        tc::tmem_relinquish();
    }
    tc_sync();
    ts.setup(N);
    ts.taddr = sm.taddr + ((uint32_t)(32 * (warp & 3)) << 16);
}

// End of a CTA: MMAs still in flight (after a wait that gave up) are waited
// for once more, bounded, then the TMEM columns are freed.
__device__ __forceinline__ void hi_tc_end(HITCShared& sm, TCState& ts, int32_t* dev_err)
{
    ts.wait_next(sm);
    ts.wait_rest(sm);
    const bool bad = __syncthreads_or(ts.bad) != 0;
    if (bad && threadIdx.x == 0) atomicOr(dev_err, BD_DEV_ERR_TC_WAIT);
    tc_sync();
    if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(sm.taddr, kTCCols);
}

// The tensor-core engine of a slot (the kernel bodies of bd_hi.cuh).
struct HITCEngine {
    using Shared = HITCShared;
    TCState ts;
    __device__ __forceinline__ void begin(Shared& sm, int N, int32_t flags)
    {
        for (int e = threadIdx.x; e < 4 * kHINTSmall; e += blockDim.x) {
            sm.pos[e] = 0.0f; sm.frc[e] = 0.0f; sm.xi[e] = 0.0f;
        }
        hi_tc_begin(sm, ts, N);
        ts.stall = (flags & BD_FLAG_TEST_TC_STALL) != 0;
    }
    __device__ __forceinline__ int step(Shared& sm, const ChainDev& ch, const StepConst<float, true>& k,
                                        const LJConst<float>& kl, const StepParams& p, int N, uint32_t key,
                                        uint32_t chain, uint32_t t, bool harmonic, bool lj)
    {
        return hi_tc_step(sm, ts, ch, k, kl, p, N, key, chain, t, harmonic, lj);
    }
    __device__ __forceinline__ bool failed() const { return ts.bad; }
    __device__ __forceinline__ void end(Shared& sm, int32_t* dev_err) { hi_tc_end(sm, ts, dev_err); }
};

__global__ void __launch_bounds__(kTCThreads, kTCBlocksPerSM) hi_tc_replica_kernel(const StepParams p)
{
    extern __shared__ __align__(128) unsigned char hi_tc_smem_raw[];
    hi_replica_body<float, true, HITCEngine>(p, *reinterpret_cast<HITCShared*>(hi_tc_smem_raw));
}

__global__ void __launch_bounds__(kTCThreads, kTCBlocksPerSM) hi_tc_parent_kernel(const StepParams p)
{
    extern __shared__ __align__(128) unsigned char hi_tc_smem_raw[];
    hi_parent_body<float, true, HITCEngine>(p, *reinterpret_cast<HITCShared*>(hi_tc_smem_raw));
}

}  // namespace bdra
