// The hot kernels of replica-averaged Brownian dynamics (Sec. II).
//
// Layout. A slot (a parent or one replica) is a run of G = ceil(N / L)
// consecutive lanes of one warp; lane `seg` of the run owns beads and springs
// seg*L .. seg*L + L-1 and keeps those L bond vectors in registers for the
// whole launch. A warp holds P = floor(32 / G) slots. Springs on the
// neighbouring lanes are reached with warp shuffles, so a step touches neither
// shared nor global memory.
//
// Two kernels share one step routine (step_bonds; collapsed chains: step_bonds_lj):
//   parent_kernel  advances every parent, writes its conformation at each
//                  window end (the "halted parent" that the next window's
//                  replicas copy; bd_set_positions writes the first), and
//                  samples it every step (ISF criteria, TSF sums); few
//                  parents run on parent_block_kernel instead;
//   replica_persist_kernel (bd_persist.cuh): warps claim (chain, replica
//                  group) items over runs of windows and evolve their replicas
//                  window after window: spawn from the parent snapshot, S
//                  steps, one force sample per replica at the window end,
//                  float64 cross-replica sum.
// The parent never reads replica state, so integrating it ahead of its
// replicas leaves every result unchanged; the noise is keyed by
// (bead, slot, step, chain), not by launch order.
//
// Bond form of Eq. 1. With free draining (Eq. 2) the update of bead i is
//   r_i += [kappa r_i + D (F_i - F_{i-1})] dt + sqrt(2 D dt) xi_i, D = 1/4,
// so the bond Q_i = r_{i+1} - r_i obeys, exactly,
//   Q_i += [kappa Q_i + D (F_{i+1} - 2 F_i + F_{i-1})] dt
//          + sqrt(2 D dt) (xi_{i+1} - xi_i),
// with F_{-1} = F_{N-1} = 0. The centre of mass, on which no force acts in a
// free-draining chain, is not carried: positions are reported in the
// centre-of-mass frame, and float32 bonds keep full relative precision however
// far a chain drifts or stretches.
//
// These units are compiled with -fmad=false: every fused multiply-add is an
// explicit fma(), so the arithmetic of a step is the same sequence of
// roundings in both kernels and for every tile size L.
#pragma once

#include "bd_conf.cuh"
#include "bd_lj.cuh"
#include "bd_step.cuh"

namespace bdra {

// ---------------------------------------------------------------------------
// Replicas, one warp work item (one replica per lane run). Lane run s of the
// warp is replica rep_begin + stride s + 1; state of replica k lives at
// state[(state_off + k (N-1)) * 3 ...]. Snapshots: snap[((w % win_ring) * M +
// spr_off + i) * 3 + d], written by the parent kernel at the end of the
// window before. wsm: this warp's scratch of kWarpScratch values.
// ---------------------------------------------------------------------------
constexpr int kWarpScratch = 512;   // >= slots per warp x springs = P (N-1) <= 32 L

// Eq. 5 diagnostics of a work item's replicas (one per lane run) at the end
// of window w; their bonds were just stored at state_slot (base of the lane's
// replica in the warp's scratch: the windows of a launch run side by side, so
// the replica's place in the state is not free for it).
template <typename T, int L>
__device__ __noinline__ void conformation_item(const ItemDev& it, const ChainDev& ch,
                                               const StepParams& p, int w, const T* state_slot,
                                               int sw, int P, int G, int bead0, bool active,
                                               int kglob)
{
    const SlotRun r = slot_run((int)(threadIdx.x & 31), sw, P, G);
    const T* pc = reinterpret_cast<const T*>(p.snap) + ((int64_t)(w % p.win_ring) * p.M + ch.spr_off) * 3;
    T acc[L][3];
#pragma unroll
    for (int j = 0; j < L; ++j) acc[j][0] = acc[j][1] = acc[j][2] = T(0);
    eq5_replica<T, L>(state_slot, pc, bead0, r, ch.N, active, acc,
                      p.dbar + ((int64_t)w * p.n_rep + ch.rep_off + kglob - 1) * 3);
    if (it.group == 0)
        eq5_rgz<T, L>(pc, bead0, r, ch.N, sw == 0, p.rgz + (int64_t)w * p.n_chains + it.chain);
    eq5_beads_out<T, L>(acc, bead0, r, sw, P, ch.N, it.rep_count,
                     p.dbead_part + ((int64_t)(w % p.win_ring) * p.bpart_stride + ch.bpart_off +
                                     (int64_t)it.group * ch.N) * 3);
}

// Window end: float64 sum over this warp's replicas of each spring's force,
// in replica order, one partial per (window, spring, group).
template <typename T>
__device__ __forceinline__ void warp_window_sum(const T* wsm, int nb, int count, double* prow)
{
    __syncwarp();
    for (int i = (int)(threadIdx.x & 31); i < nb; i += 32) {
        double acc = 0.0;
        for (int s = 0; s < count; ++s) acc += (double)wsm[s * nb + i];
        prow[i] = acc;
    }
    __syncwarp();
}

// The same samples a row a replica (ChainDev::own_per_warp); prow: replica 0's.
template <typename T>
__device__ __forceinline__ void warp_window_rows(const T* wsm, int nb, const ItemDev& it, double* prow)
{
    __syncwarp();
    for (int s = 0; s < it.rep_count; ++s)
        for (int i = (int)(threadIdx.x & 31); i < nb; i += 32)
            prow[(int64_t)(it.rep_begin + it.stride * s) * nb + i] = (double)wsm[s * nb + i];
    __syncwarp();
}

// With TAB, ptab is this warp's table of 32 L bead parts of the Philox
// counter (filled here for the item's chain). CONF compiles in the Eq. 5
// window-end diagnostics (used when BD_FLAG_CONFORMATION is set); without it
// the step loop carries no trace of them. H: the noise half of every replica
// of the item (known when all are odd or all even), or -1.
template <typename T, int L, bool FAST, bool TAB, bool CONF, bool LJ, int H>
__device__ __forceinline__ void run_one_item_h(const ItemDev& it, const StepRange& rg, const StepParams& p,
                                               T* wsm, uint4* ptab, T* conf)
{
    const ChainDev ch = p.chains[it.chain];
    const int nb = ch.N - 1;
    const int G = (ch.N + L - 1) / L;
    const int P = 32 / G;
    const int lane = threadIdx.x & 31;
    const int sw = lane / G;
    const bool active = (sw < P) && (sw < it.rep_count);
    const int kglob = it.rep_begin + it.stride * sw + 1;
    const uint32_t key = (p.flags & BD_FLAG_IDENTICAL_NOISE) ? 0u : (uint32_t)kglob;
    const LaneCtx lc = make_lane(sw < P ? lane - sw * G : 0, G, L, lane, nb, active, key,
                                 (uint32_t)it.chain + p.chain_base);
    StepConst<T, FAST> k;
    k.load(ch, p);
    LJConst<T> kl;
    if (LJ) kl.load(ch);
    if (TAB) {
        for (int b = lane; b < G * L; b += 32)
            ptab[b] = PhiloxSplit::bead_part((uint32_t)b, (uint32_t)it.chain + p.chain_base, p.rk0, p.rk1);
        __syncwarp();
    }

    T* state = reinterpret_cast<T*>(p.state) + (ch.state_off + (int64_t)kglob * nb) * 3;
    const T* snap = reinterpret_cast<const T*>(p.snap);
    T qx[L], qy[L], qz[L];
    // the replica's state where the launch starts inside a window, else the
    // snapshot (one load from either place: a branch around it cost 12 registers
    // on the 4-spring tile); a part after the first never reads the state that
    // the last one writes
    load_bonds<T, L>(qx, qy, qz, rg.s_in != 0 ? state : snap + ((int64_t)(rg.w % p.win_ring) * p.M + ch.spr_off) * 3, lc);

    int floored = 0;
    int s_in = rg.s_in;
    int w = rg.w;                                   // window index (< 2^31)
#pragma unroll 1
    for (uint32_t t = rg.t0; t < rg.t1; ++t) {
        if (s_in == 0 && t != rg.t0)   // spawn: copy the halted parent (Sec. II)
            load_bonds<T, L>(qx, qy, qz, snap + ((int64_t)(w % p.win_ring) * p.M + ch.spr_off) * 3, lc);
        if constexpr (LJ)
            floored += step_bonds_lj<T, L, FAST, TAB, H>(qx, qy, qz, lc, k, kl, sw < P, sw < P ? lane - sw * G : 0, G,
                                           sw < P ? sw * G : lane, (uint32_t)t, p, ptab);
        else
            floored += step_bonds<T, L, FAST, TAB, H>(qx, qy, qz, lc, k, (uint32_t)t, p, ptab);
        if (++s_in == p.S) {
            // one force sample per replica at the end of the evolution time
            s_in = 0;
            if (active) {
#pragma unroll
                for (int j = 0; j < L; ++j) {
                    const int i = lc.bead0 + j;
                    if (i < nb)
                        wsm[sw * nb + i] =
                            LJ ? rest_law_tension<T, FAST>(qx[j], qy[j], qz[j], (i & 1) == 0, k.H, kl, k.smin)
                               : spring_tension<T, FAST>(qx[j], qy[j], qz[j], k.H, k.Hinvb, k.smin);
                }
            }
            double* prow = p.part_hist + (int64_t)(w % p.win_ring) * p.part_stride + ch.part_off;
            if (sizeof(T) == 8 && !LJ && !CONF && ch.own_per_warp > 0) warp_window_rows<T>(wsm, nb, it, prow);
            else warp_window_sum<T>(wsm, nb, it.rep_count, prow + (int64_t)it.group * nb);
            if (CONF && (p.flags & BD_FLAG_CONFORMATION)) {
                T* mine = conf + (sw < P ? sw : 0) * nb * 3;
                store_bonds<T, L>(qx, qy, qz, mine, lc);
                conformation_item<T, L>(it, ch, p, w, mine, sw, P, G, lc.bead0, active, kglob);
            }
            ++w;
        }
    }
    if (rg.last) store_bonds<T, L>(qx, qy, qz, state, lc);
    if (floored) atomicAdd(p.overext + it.chain, (unsigned long long)floored);
    if (TAB) __syncwarp();     // every lane is done with ptab before the next item refills it
}

// A work item with one replica per lane run. The planner gives such an item
// only odd or only even replicas (stride 2) or a single one, so all its
// replicas draw the same half of their noise pairs' generator outputs (in
// identical-noise runs all draw the parent's, half 0): the half is fixed
// for the whole warp and compiled in.
template <typename T, int L, bool FAST, bool TAB = false, bool CONF = false, bool LJ = false>
__device__ __forceinline__ void run_one_item(const ItemDev& it, const StepRange& rg, const StepParams& p, T* wsm,
                                             uint4* ptab, T* conf)
{
    const bool h1 = (p.flags & BD_FLAG_IDENTICAL_NOISE) == 0 && noise_half((uint32_t)it.rep_begin + 1u) == 1u;
    if (h1) run_one_item_h<T, L, FAST, TAB, CONF, LJ, 1>(it, rg, p, wsm, ptab, conf);
    else run_one_item_h<T, L, FAST, TAB, CONF, LJ, 0>(it, rg, p, wsm, ptab, conf);
}

// ---------------------------------------------------------------------------
// Few parents of Hooke and FENE chains. CTA g holds parent_warps[g].count parents
// (chains parent_items[first + s]), each on G lanes of warp 0.
//
// A parent's steps are a serial chain, and the one warp of parent_kernel that
// draws the noise, takes the step and samples it issues about 620
// instructions a step (4-spring tile) at the rate of a lone warp: 1.1-1.3 us
// a step in float32, 4.8 us in float64. Only the forces and the update depend on the
// state, so the rest moves to the CTA's other warps, B steps at a time: warp
// 0 takes the steps of block k from the noise in shared memory and leaves the
// bonds of every step there, while warps 1..3 draw the noise of block k + 1
// and sample the bonds of block k - 1 (TSF sums, ISF criteria; the springs
// of a helper thread stay with it, so every sum keeps its order). One CTA
// barrier a block. The rounding sequence is that of step_bonds: the helpers
// store the difference of the two beads' normals that the update would form.
// It issues more in all (idle helper lanes, the buffers), so many parents,
// which fill the GPU anyway, stay with parent_kernel (bd_api.cu:
// kParentBlockWarps).
// ---------------------------------------------------------------------------
template <typename T, int L> struct ParentBlock {
    static constexpr int helpers = kParentThreads2 - 32;
    static constexpr int E = 32 * L;                            // springs (and beads) of the CTA
    static constexpr int B = L <= 4 ? 8 : L <= 7 ? 4 : L <= 10 ? 3 : 2;   // steps a block (48 KB of buffers in float32)
    static constexpr int NS = (E + helpers - 1) / helpers;      // springs a helper samples
    static constexpr int rows = 2 * B * 3;                      // rows of E values of each buffer
    struct Chain {                                              // sampling constants of one parent
        T H, Hinvb, smin, fc;
        BellConst bell;
        int64_t spr_off;
        int32_t nb, pad;
    };
    static constexpr size_t bytes = sizeof(uint4) * E + sizeof(Chain) * 32 + sizeof(T) * 2 * rows * E;
};

// A lane's L values of a row (value lane L + j), in the widest loads that L allows.
template <typename T, int L>
__device__ __forceinline__ void row_load(const T* row, int lane, T (&v)[L])
{
    constexpr int W = sizeof(T) == 4 ? (L % 4 == 0 ? 4 : L % 2 == 0 ? 2 : 1) : (L % 2 == 0 ? 2 : 1);
    struct alignas(sizeof(T) * W) Vec { T e[W]; };
    const Vec* src = reinterpret_cast<const Vec*>(row + lane * L);
#pragma unroll
    for (int j = 0; j < L / W; ++j) {
        const Vec x = src[j];
#pragma unroll
        for (int e = 0; e < W; ++e) v[W * j + e] = x.e[e];
    }
}
template <typename T, int L>
__device__ __forceinline__ void row_store(T* row, int lane, const T (&v)[L])
{
    constexpr int W = sizeof(T) == 4 ? (L % 4 == 0 ? 4 : L % 2 == 0 ? 2 : 1) : (L % 2 == 0 ? 2 : 1);
    struct alignas(sizeof(T) * W) Vec { T e[W]; };
    Vec* dst = reinterpret_cast<Vec*>(row + lane * L);
#pragma unroll
    for (int j = 0; j < L / W; ++j) {
        Vec x;
#pragma unroll
        for (int e = 0; e < W; ++e) x.e[e] = v[W * j + e];
        dst[j] = x;
    }
}

// step_bonds with the noise differences xi_{i+1} - xi_i of the lane's springs
// given (the same rounding sequence).
template <typename T, int L, bool FAST>
__device__ __forceinline__ int step_bonds_given(T (&qx)[L], T (&qy)[L], T (&qz)[L], const T (&dx)[L],
                                                const T (&dy)[L], const T (&dz)[L], const LaneCtx& lc,
                                                const StepConst<T, FAST>& k)
{
    int fl = 0;
    T fx[L], fy[L], fz[L];
#pragma unroll
    for (int j = 0; j < L; ++j) {
        const T c = spring_coef<T, FAST>(qx[j], qy[j], qz[j], k.H, k.Hinvb, k.smin, fl);
        fx[j] = c * qx[j]; fy[j] = c * qy[j]; fz[j] = c * qz[j];
    }
    T fmx = shfl(fx[L - 1], lc.src_prev), fmy = shfl(fy[L - 1], lc.src_prev), fmz = shfl(fz[L - 1], lc.src_prev);
    T fnx = shfl(fx[0], lc.src_next), fny = shfl(fy[0], lc.src_next), fnz = shfl(fz[0], lc.src_next);
    if (!lc.has_prev) { fmx = T(0); fmy = T(0); fmz = T(0); }
    if (!lc.has_next) { fnx = T(0); fny = T(0); fnz = T(0); }
#pragma unroll
    for (int j = 0; j < L; ++j) {
        const T px = j + 1 < L ? fx[j + 1 < L ? j + 1 : 0] : fnx;
        const T py = j + 1 < L ? fy[j + 1 < L ? j + 1 : 0] : fny;
        const T pz = j + 1 < L ? fz[j + 1 < L ? j + 1 : 0] : fnz;
        if (j < lc.nv) {
            const T lx = fma(T(-2), fx[j], px + fmx);
            const T ly = fma(T(-2), fy[j], py + fmy);
            const T lz = fma(T(-2), fz[j], pz + fmz);
            const T ox = qx[j], oy = qy[j], oz = qz[j];
            qx[j] = fma(k.cn, dx[j], fma(k.cd, lx, fma(k.axz, oz, fma(k.axx, ox, ox))));
            qy[j] = fma(k.cn, dy[j], fma(k.cd, ly, fma(k.ayy, oy, oy)));
            qz[j] = fma(k.cn, dz[j], fma(k.cd, lz, fma(k.azz, oz, oz)));
        }
        fmx = fx[j]; fmy = fy[j]; fmz = fz[j];
    }
    return lc.active ? fl : 0;
}

// The CTA's barrier between blocks, met by its warps in different code.
__device__ __forceinline__ void parent_barrier()
{
    asm volatile("bar.sync 1, %0;" :: "n"(kParentThreads2) : "memory");
}

template <typename T, int L, bool FAST>
__global__ void __launch_bounds__(kParentThreads2)
parent_block_kernel(const StepParams p)
{
    using PB = ParentBlock<T, L>;
    constexpr int E = PB::E, B = PB::B, NS = PB::NS;
    extern __shared__ uint4 bd_parent_smem[];
    uint4* ptab = bd_parent_smem;                                        // Philox bead parts, parent s at [s G L, (s + 1) G L)
    T* noise = reinterpret_cast<T*>(ptab + E);                           // [2][B][3][E]
    T* bonds = noise + PB::rows * E;                                     // [2][B][3][E]
    typename PB::Chain* pc = reinterpret_cast<typename PB::Chain*>(bonds + PB::rows * E);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const ParentWarp pw = p.parent_warps[blockIdx.x];
    const int G = pw.G, P = 32 / G, GL = G * L, beads = P * GL;
    const int64_t M = p.M;
    for (int e = threadIdx.x; e < beads; e += blockDim.x) {
        const int s = e / GL;
        const int c = p.parent_items[pw.first + min(s, pw.count - 1)];
        ptab[e] = PhiloxSplit::bead_part((uint32_t)(e - s * GL), (uint32_t)c + p.chain_base, p.rk0, p.rk1);
    }
    if ((int)threadIdx.x < pw.count) {
        const ChainDev& ch = p.chains[p.parent_items[pw.first + threadIdx.x]];
        StepConst<T, FAST> k;
        k.load(ch, p);
        typename PB::Chain& o = pc[threadIdx.x];
        o.H = k.H; o.Hinvb = k.Hinvb; o.smin = k.smin;
        o.fc = (T)ch.f_c;
        o.bell.load(ch.k0, p.dt, ch.dx);
        o.spr_off = ch.spr_off;
        o.nb = ch.N - 1;
    }
    __syncthreads();

    const int64_t nblk = (p.n_steps + B - 1) / B;
    if (warp == 0) {
        // the integrator: wait for the noise of block k, take its steps
        const int sw = lane / G;
        const bool active = sw < P && sw < pw.count;
        const int c = p.parent_items[pw.first + (active ? sw : 0)];
        const ChainDev& ch = p.chains[c];
        const int64_t spr_off = ch.spr_off;
        const LaneCtx lc = make_lane(sw < P ? lane - sw * G : 0, G, L, lane, ch.N - 1, active, 0u, (uint32_t)c + p.chain_base);
        StepConst<T, FAST> k;
        k.load(ch, p);
        T* state = reinterpret_cast<T*>(p.state) + ch.state_off * 3;
        T* snap = reinterpret_cast<T*>(p.snap);
        T qx[L], qy[L], qz[L];
        load_bonds<T, L>(qx, qy, qz, state, lc);
        int floored = 0;
        int s_in = (int)(p.t0 % p.S);
        int64_t w = p.t0 / p.S, left = p.n_steps;
        for (int64_t b = 0; b <= nblk; ++b) {
            parent_barrier();
            const int nb_steps = left < B ? (int)left : B;
            left -= nb_steps;
            T* nrow = noise + (b & 1) * (B * 3 * E);
            T* brow = bonds + (b & 1) * (B * 3 * E);
#pragma unroll 1
            for (int s = 0; s < nb_steps; ++s, nrow += 3 * E, brow += 3 * E) {
                T dx[L], dy[L], dz[L];
                row_load<T, L>(nrow, lane, dx);
                row_load<T, L>(nrow + E, lane, dy);
                row_load<T, L>(nrow + 2 * E, lane, dz);
                floored += step_bonds_given<T, L, FAST>(qx, qy, qz, dx, dy, dz, lc, k);
                row_store<T, L>(brow, lane, qx);
                row_store<T, L>(brow + E, lane, qy);
                row_store<T, L>(brow + 2 * E, lane, qz);
                if (++s_in == p.S) {   // the conformation the replicas of the next window start from
                    s_in = 0;
                    ++w;
                    store_bonds<T, L>(qx, qy, qz, snap + ((w % p.win_ring) * M + spr_off) * 3, lc);
                }
            }
        }
        store_bonds<T, L>(qx, qy, qz, state, lc);
        if (floored) atomicAdd(p.overext + c, (unsigned long long)floored);
        return;
    }

    // helpers: noise of the block ahead, samples of the block behind. A
    // noise unit is one step of 31 springs (32 beads); a helper thread samples
    // springs h + 96 j of the CTA.
    const int h = (int)threadIdx.x - 32;
    const bool isf_thr = (p.thr_mask & BD_CRIT_ISF) != 0;
    const bool isf_bell = (p.bell_mask & BD_CRIT_ISF) != 0;
    ParentSums<T> sums[NS];
    uint32_t mine = 0, thr_done = 0, bell_done = 0;
    int par[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const int e = h + PB::helpers * j, s = e / GL;
        const bool v = s < P && s < pw.count && e - s * GL < pc[s < pw.count ? s : 0].nb;
        par[j] = v ? s : 0;
        const int64_t m = v ? pc[s].spr_off + (e - s * GL) : 0;
        sums[j].start(v ? p.tsf_acc[m] : 0.0, v ? p.exp1[CRIT_Q_ISF * M + m] - p.lam[CRIT_Q_ISF * M + m] : 0.0);
        if (v) mine |= 1u << j;
        if (!v || p.first_thr[CRIT_Q_ISF * M + m] >= 0) thr_done |= 1u << j;
        if (!v || p.first_bell[CRIT_Q_ISF * M + m] >= 0) bell_done |= 1u << j;
    }
    const int chunks = (beads + 30) / 31;
    int s_in = (int)(p.t0 % p.S);
    int64_t w = p.t0 / p.S;
    for (int64_t b = -1; b <= nblk; ++b) {
        if (b + 1 < nblk) {                                     // noise of block b + 1
            const int64_t t_b = p.t0 + (b + 1) * B;
            const int steps = p.t0 + p.n_steps - t_b < B ? (int)(p.t0 + p.n_steps - t_b) : B;
            T* nb0 = noise + ((b + 1) & 1) * (B * 3 * E);
            for (int u = warp - 1; u < steps * chunks; u += PB::helpers / 32) {
                const int s = u / chunks, e = (u - s * chunks) * 31 + lane;
                const uint3 sp = PhiloxSplit::step_part((uint32_t)(t_b + s), noise_word(0u), p.rk0);
                T z0, z1, z2;
                bead_noise_split<T, FAST, 0>(ptab[min(e, beads - 1)], sp, p, 0u, z0, z1, z2);
                const T y0 = __shfl_down_sync(0xffffffffu, z0, 1), y1 = __shfl_down_sync(0xffffffffu, z1, 1),
                        y2 = __shfl_down_sync(0xffffffffu, z2, 1);
                if (lane < 31 && e < beads) {
                    T* row = nb0 + s * 3 * E + e;
                    row[0] = y0 - z0;
                    row[E] = y1 - z1;
                    row[2 * E] = y2 - z2;
                }
            }
        }
        if (b >= 1) {                                           // samples of block b - 1
            const int64_t t_b = p.t0 + (b - 1) * B;
            const int steps = p.t0 + p.n_steps - t_b < B ? (int)(p.t0 + p.n_steps - t_b) : B;
            const T* brow = bonds + ((b - 1) & 1) * (B * 3 * E) + h;
#pragma unroll 1
            for (int s = 0; s < steps; ++s, brow += 3 * E) {
                const bool ends = ++s_in == p.S;
#pragma unroll
                for (int j = 0; j < NS; ++j) {
                    if (!(mine & (1u << j))) continue;
                    const typename PB::Chain& o = pc[par[j]];
                    const int d = PB::helpers * j;
                    const T f = spring_tension<T, FAST>(brow[d], brow[E + d], brow[2 * E + d], o.H, o.Hinvb, o.smin);
                    sums[j].add_isf(f);
                    const int64_t m = o.spr_off + (h + d - par[j] * GL);
                    if (isf_thr && !(thr_done & (1u << j)) && f >= o.fc) {
                        thr_done |= 1u << j;
                        p.first_thr[CRIT_Q_ISF * M + m] = t_b + s + 1;
                    }
                    if (isf_bell) {
                        const bool reached = sums[j].add_hazard(f, o.bell, p.lam + CRIT_Q_ISF * M + m);
                        if (!(bell_done & (1u << j)) && reached) {
                            bell_done |= 1u << j;
                            p.first_bell[CRIT_Q_ISF * M + m] = t_b + s + 1;
                        }
                    }
                    if (ends) {
                        p.tsf_hist[w * M + m] = sums[j].tsf_sum() / (double)p.S;
                        double rem = 0.0;
                        if (isf_bell) {
                            const double lam = p.lam[CRIT_Q_ISF * M + m] + sums[j].hazard();
                            p.lam[CRIT_Q_ISF * M + m] = lam;
                            rem = p.exp1[CRIT_Q_ISF * M + m] - lam;
                        }
                        sums[j].next_window(rem);
                    }
                }
                if (ends) { s_in = 0; ++w; }
            }
        }
        if (b < nblk) parent_barrier();
    }
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        if (!(mine & (1u << j))) continue;
        const int64_t m = pc[par[j]].spr_off + (h + PB::helpers * j - par[j] * GL);
        p.tsf_acc[m] = sums[j].tsf_sum();
        if (isf_bell) p.lam[CRIT_Q_ISF * M + m] += sums[j].hazard();
    }
}

// ---------------------------------------------------------------------------
// Parents. Global warp g holds parent_warps[g].count parents (chains
// parent_items[first + s]), each on G lanes.
// Per step: update, then sample the parent's spring forces (ISF): TSF window
// sums and ISF threshold / Bell criteria. Window sums and the window's hazard
// stay in registers; the integrated hazard lives in p.lam (float64).
// ---------------------------------------------------------------------------
template <typename T, int L, bool FAST, bool LJ = false>
__global__ void __launch_bounds__(kParentThreads)
parent_kernel(const StepParams p)
{
    // per warp: the split-Philox bead parts of its parents' beads, parent s
    // at [s G L, (s + 1) G L)
    __shared__ uint4 ptab_all[kParentThreads / 32][32 * L];
    const int lane = threadIdx.x & 31;
    if ((int)(threadIdx.x >> 5) >= kParentThreads / 32) return;   // whole warps beyond the table
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (gw >= p.n_parent_warps) return;          // whole warp: no shuffle partner left behind
    const ParentWarp pw = p.parent_warps[gw];
    const int G = pw.G;
    const int P = 32 / G;
    const int sw = lane / G;
    const bool active = (sw < P) && (sw < pw.count);
    const int c = p.parent_items[pw.first + (active ? sw : 0)];
    const ChainDev ch = p.chains[c];
    const int nb = ch.N - 1;
    const LaneCtx lc = make_lane(sw < P ? lane - sw * G : 0, G, L, lane, nb, active, 0u,
                                 (uint32_t)c + p.chain_base);
    StepConst<T, FAST> k;
    k.load(ch, p);
    LJConst<T> kl;
    if (LJ) kl.load(ch);
    uint4* ptab = ptab_all[threadIdx.x >> 5];
    for (int e = lane; e < P * G * L; e += 32) {
        const int s2 = e / (G * L);
        const int c2 = p.parent_items[pw.first + min(s2, pw.count - 1)];
        ptab[e] = PhiloxSplit::bead_part((uint32_t)(e - s2 * G * L), (uint32_t)c2 + p.chain_base, p.rk0, p.rk1);
    }
    __syncwarp();
    const uint4* my_tab = ptab + (sw < P ? sw : 0) * G * L;
    const int64_t M = p.M;
    const bool isf_thr = (p.thr_mask & BD_CRIT_ISF) != 0;
    const bool isf_bell = (p.bell_mask & BD_CRIT_ISF) != 0;
    const T fc = (T)ch.f_c;
    BellConst bk;
    bk.load(ch.k0, p.dt, ch.dx);

    T* state = reinterpret_cast<T*>(p.state) + ch.state_off * 3;
    T* snap = reinterpret_cast<T*>(p.snap);
    T qx[L], qy[L], qz[L];
    load_bonds<T, L>(qx, qy, qz, state, lc);

    // per-spring sampling state of this lane's springs: the time-average sum
    // and the Bell hazard in float64, or float-float pairs with float32
    // integration (a plain float32 sum over a 1500-step window would lose
    // about three digits of the TSF before the division)
    ParentSums<T> sums[L];
    // quiet: springs outside the criteria (the disulfide bonds of a vWF chain)
    uint32_t thr_done = 0, bell_done = 0, quiet = 0;
#pragma unroll
    for (int j = 0; j < L; ++j) {
        const int i = lc.bead0 + j;
        const int64_t m = ch.spr_off + i;
        const bool v = active && i < nb;
        sums[j].start(v ? p.tsf_acc[m] : 0.0, v ? p.exp1[CRIT_Q_ISF * M + m] - p.lam[CRIT_Q_ISF * M + m] : 0.0);
        if (ch.spring == BD_SPRING_VWF && (i & 1)) quiet |= 1u << j;
        if (!v || p.first_thr[CRIT_Q_ISF * M + m] >= 0) thr_done |= 1u << j;
        if (!v || p.first_bell[CRIT_Q_ISF * M + m] >= 0) bell_done |= 1u << j;
    }
    thr_done |= quiet;
    bell_done |= quiet;

    int floored = 0;
    int s_in = (int)(p.t0 % p.S);
    int64_t w = p.t0 / p.S;
    const int64_t t_end = p.t0 + p.n_steps;
#pragma unroll 1
    for (int64_t t = p.t0; t < t_end; ++t) {
        if constexpr (LJ)
            floored += step_bonds_lj<T, L, FAST, true, 0>(qx, qy, qz, lc, k, kl, sw < P, sw < P ? lane - sw * G : 0, G,
                                            sw < P ? sw * G : lane, (uint32_t)t, p, my_tab);
        else
            floored += step_bonds<T, L, FAST, true, 0>(qx, qy, qz, lc, k, (uint32_t)t, p, my_tab);
        if (active) {
#pragma unroll
            for (int j = 0; j < L; ++j) {
                const int i = lc.bead0 + j;
                if (i < nb) {
                    const T f = LJ ? rest_law_tension<T, FAST>(qx[j], qy[j], qz[j], (i & 1) == 0, k.H, kl, k.smin)
                                   : spring_tension<T, FAST>(qx[j], qy[j], qz[j], k.H, k.Hinvb, k.smin);
                    sums[j].add_isf(f);
                    if (isf_thr && !(thr_done & (1u << j)) && f >= fc) {
                        thr_done |= 1u << j;
                        p.first_thr[CRIT_Q_ISF * M + ch.spr_off + i] = t + 1;
                    }
                    if (isf_bell && !(quiet & (1u << j))) {
                        const bool reached = sums[j].add_hazard(f, bk, p.lam + CRIT_Q_ISF * M + ch.spr_off + i);
                        if (!(bell_done & (1u << j)) && reached) {
                            bell_done |= 1u << j;
                            p.first_bell[CRIT_Q_ISF * M + ch.spr_off + i] = t + 1;
                        }
                    }
                }
            }
        }
        if (++s_in == p.S) {
            s_in = 0;
            if (active) {
#pragma unroll
                for (int j = 0; j < L; ++j) {
                    const int i = lc.bead0 + j;
                    if (i < nb) {
                        const int64_t m = ch.spr_off + i;
                        p.tsf_hist[w * M + m] = sums[j].tsf_sum() / (double)p.S;
                        double rem = 0.0;
                        if (isf_bell) {
                            const double lam = p.lam[CRIT_Q_ISF * M + m] + sums[j].hazard();
                            p.lam[CRIT_Q_ISF * M + m] = lam;
                            rem = p.exp1[CRIT_Q_ISF * M + m] - lam;
                        }
                        sums[j].next_window(rem);
                    }
                }
            }
            ++w;
            // the conformation the replicas of the next window start from
            store_bonds<T, L>(qx, qy, qz, snap + ((w % p.win_ring) * M + ch.spr_off) * 3, lc);
        }
    }
    store_bonds<T, L>(qx, qy, qz, state, lc);
    if (active) {
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const int i = lc.bead0 + j;
            if (i < nb) {
                const int64_t m = ch.spr_off + i;
                p.tsf_acc[m] = sums[j].tsf_sum();
                if (isf_bell) p.lam[CRIT_Q_ISF * M + m] += sums[j].hazard();
            }
        }
    }
    if (floored) atomicAdd(p.overext + c, (unsigned long long)floored);
}

}  // namespace bdra
