// orca_cluster_bin.cuh -- the binning step of small scenes as one
// thread-block cluster (sm_103a).
//
// bin_kernel sorts the agents through global memory in phases separated by
// grid barriers; with few agents each phase is a few dependent L2 round trips
// and a barrier, 16 us a step however small the scene.  Here the cell counts,
// the cell starts and the cell-order records live in the shared memory of at
// most 16 blocks of one cluster: block r owns a contiguous range of cells and
// a contiguous range of slots, the others reach them through distributed
// shared memory, and the hardware cluster barrier (every block of a cluster is
// resident) separates the phases.  The sorted state is the same as
// bin_kernel's up to the order of agents with equal cell and x, which no
// result depends on.
#pragma once

#include <cooperative_groups.h>

#include "orca_step_kernels.cuh"

namespace orca {

constexpr int kClusterMax = 16;
constexpr int kClusterThreads = 1024;
constexpr int kClusterPerThread = 2;                                 // agents
constexpr int kClusterSlots = kClusterThreads * kClusterPerThread;   // per block
constexpr int kClusterCells = 32768;                                 // per block

constexpr int kClusterThreadsFew = 512;    // threads of a block in scenes of few agents
constexpr int kClusterCellsFew = 4096;     // and few cells

// log2 sizes of the cell and slot ranges of a block, and its threads
struct ClusterShape {
    int cell_shift;
    int slot_shift;
    int threads;
};

inline size_t cluster_smem(ClusterShape sh) {
    return ((size_t)16 << sh.slot_shift) + ((size_t)4 << sh.cell_shift) + 16;
}

// The cluster barrier in two halves: what a block writes between them need not
// be visible to the others, so the barrier does not wait for it, and loads that
// need nothing from the others overlap it.  An arrival also waits until the
// block's earlier writes have reached memory (a fence: a quarter of the kernel's
// stalls with whole barriers), so global writes stand behind it.  1.1 us a step
// (4,064 agents, 16 steps and their gradient 676 -> 650 us; 16,250 agents, 4 steps
// 193 -> 189).  Every thread of every block calls both.
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <class SRC, bool FIRST, int NT>
__global__ void __launch_bounds__(NT)
cluster_bin_kernel(SRC src, BinArgs a, ClusterShape sh) {
    namespace cg = cooperative_groups;
    extern __shared__ uint4 cluster_mem[];
    __shared__ uint32_t ws[32], total, base[kClusterMax + 1];
    const cg::cluster_group cl = cg::this_cluster();
    const int r = (int)blockIdx.x, nb = (int)gridDim.x, tid = (int)threadIdx.x;
    const int cn = 1 << sh.cell_shift, sn = 1 << sh.slot_shift;
    uint4* slots = cluster_mem;                                    // sn cell-order records
    uint32_t* cells = reinterpret_cast<uint32_t*>(slots + sn);     // cn counts, later starts

    // the solve kernel may be set up meanwhile; what ran before is finished
    // before any state is read
    launch_dependents();
    for (int q = tid; q <= cn; q += NT) cells[q] = 0u;
    cluster_arrive();
    wait_for_primary();

    // ---- the agents of this block and their cells ----
    // (first step: in the order that the previous call recorded, if it did, so
    // that a block's agents lie in few blocks' cells)
    const uint32_t* hint = nullptr;
    if (FIRST && __ldcg(a.err + 1) != 0) hint = a.hint;
    const int i0 = r << sh.slot_shift;
    const int iend = min(i0 + sn, a.n);
    int from[kClusterPerThread];
    float x[kClusterPerThread];
    uint32_t c[kClusterPerThread];
    bool bad = false, lost = false;
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        from[u] = i0 + tid + u * NT;
        if (FIRST && hint != nullptr && from[u] < iend) {
            const uint32_t h = hint[from[u]];
            if (h < (uint32_t)a.n) from[u] = (int)h;
            else lost = true;
        }
    }
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        c[u] = 0xffffffffu;
        x[u] = 0.0f;
        if (i0 + tid + u * NT < iend) {
            const int i = from[u];
            const float2 p = FIRST ? a.upos[i] : a.pos0[i];
            if (FIRST) {
                const float2 v = a.uvel[i];
                bad |= !(isfinite(p.x) && isfinite(p.y) && isfinite(v.x) && isfinite(v.y));
            }
            const SceneDev& sc = src.get(i);
            x[u] = p.x;
            c[u] = (uint32_t)(sc.cell_off +
                              cell_axis(p.y, sc.origin_y, sc.inv_cell_y, sc.ny) * sc.nx +
                              cell_axis(p.x, sc.origin_x, sc.inv_cell_x, sc.nx));
        }
    }
    if (lost) atomicOr(a.err, ERR_BIT_STATE);
    if (bad) atomicOr(a.err, ERR_BIT_NONFINITE);
    cluster_wait();   // every block's counts are zero

    // ---- counting ----
    uint32_t slot[kClusterPerThread];
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        slot[u] = 0u;
        if (c[u] != 0xffffffffu) {
            uint32_t* rc = cl.map_shared_rank(cells, (unsigned)(c[u] >> sh.cell_shift));
            slot[u] = atomicAdd(rc + (c[u] & (uint32_t)(cn - 1)), 1u);
        }
    }
    cluster_arrive();
    cluster_wait();

    // ---- starts within the block's cells, and the blocks' totals ----
    {
        uint32_t carry = 0u;
        for (int q0 = 0; q0 < cn; q0 += 4 * NT) {
            const int q = q0 + 4 * tid;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (q < cn) v = *reinterpret_cast<const uint4*>(cells + q);
            uint32_t tile;
            const uint32_t o = carry + block_excl_scan(v.x + v.y + v.z + v.w, ws, tile);
            if (q < cn)
                *reinterpret_cast<uint4*>(cells + q) =
                    make_uint4(o, o + v.x, o + v.x + v.y, o + v.x + v.y + v.z);
            carry += tile;
        }
        if (tid == 0) {
            cells[cn] = carry;
            total = carry;
        }
    }
    cluster_arrive();
    cluster_wait();
    if (tid < 32) {
        uint32_t t = tid < nb ? *cl.map_shared_rank(&total, (unsigned)tid) : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (tid >= o) t += y;
        }
        if (tid < nb) base[tid + 1] = t;
        if (tid == 0) base[0] = 0u;
    }
    __syncthreads();

    // ---- records into cell order; the starts for the search ----
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        if (c[u] != 0xffffffffu) {
            const unsigned own = (unsigned)(c[u] >> sh.cell_shift);
            const uint32_t* rc = cl.map_shared_rank(cells, own) + (c[u] & (uint32_t)(cn - 1));
            const uint32_t b = base[own] + rc[0], e = base[own] + rc[1], d = b + slot[u];
            uint4* rs = cl.map_shared_rank(slots, (unsigned)(d >> sh.slot_shift));
            rs[d & (uint32_t)(sn - 1)] = make_uint4(x_order_key(x[u]), (uint32_t)from[u], b, e);
        }
    }
    cluster_arrive();
    const int c0 = r << sh.cell_shift;
    for (int q = tid; q < cn && c0 + q < a.ncells; q += NT)
        a.start[c0 + q] = base[r] + cells[q];
    if (r == nb - 1 && tid == 0) a.start[a.ncells] = (uint32_t)a.n;
    cluster_wait();

    // ---- order by x inside every cell (ties by slot); move the state ----
    float2 p[kClusterPerThread], v[kClusterPerThread];
    uint2 ax[kClusterPerThread];
    uint32_t dst[kClusterPerThread];
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        const int t = i0 + tid + u * NT;
        p[u] = v[u] = make_float2(0.0f, 0.0f);
        ax[u] = make_uint2(0u, 0u);
        dst[u] = 0u;
        if (t < iend) {
            const uint4 e = slots[t - i0];
            const uint32_t i = e.y;
            p[u] = FIRST ? a.upos[i] : a.pos0[i];
            v[u] = FIRST ? a.uvel[i] : a.vel0[i];
            ax[u] = FIRST ? aux_pack(a.urad[i], a.utype[i], (int)i) : a.aux0[i];
            uint32_t rank = 0u;
            for (uint32_t w = e.z; w < e.w; ++w) {
                const unsigned own = (unsigned)(w >> sh.slot_shift);
                const uint4* rs = own == (unsigned)r ? slots : cl.map_shared_rank(slots, own);
                const uint32_t xv = rs[w & (uint32_t)(sn - 1)].x;
                rank += (xv < e.x || (xv == e.x && w < (uint32_t)t)) ? 1u : 0u;
            }
            dst[u] = e.z + rank;
        }
    }
    cluster_arrive();
#pragma unroll
    for (int u = 0; u < kClusterPerThread; ++u) {
        if (i0 + tid + u * NT < iend) {
            a.pos1[dst[u]] = p[u];
            a.vel1[dst[u]] = v[u];
            a.aux1[dst[u]] = ax[u];
        }
    }
    cluster_wait();   // no block leaves while another reads its records
}

// ------------------------------------------------------- no cells at all ----
// The smallest scenes: the agents sorted by one coordinate (y if by_y), by
// counting for each agent the keys below its own (equal ones by index).  Every
// block reads all coordinates, so no block waits for another: one round trip to
// memory and n / 8 comparisons per lane (eight lanes an agent) in place of the
// cluster's count, scan, scatter and rank.
constexpr int kFlatMax = 1024;
constexpr int kFlatThreads = 256;
constexpr int kFlatLanes = 8;
constexpr int kFlatAgents = kFlatThreads / kFlatLanes;   // per block

template <bool FIRST>
__global__ void __launch_bounds__(kFlatThreads) flat_bin_kernel(BinArgs a, bool by_y) {
    __shared__ uint32_t keys[kFlatMax];
    launch_dependents();
    wait_for_primary();
    const float2* pos = FIRST ? a.upos : a.pos0;
    const int tid = (int)threadIdx.x, q = tid % kFlatLanes;
    const int i = (int)blockIdx.x * kFlatAgents + tid / kFlatLanes;
    float2 p = make_float2(0.0f, 0.0f), v = p;
    uint2 ax = make_uint2(0u, 0u);
    if (i < a.n) {   // (its loads overlap the staging)
        p = pos[i];
        if (q == 0) {
            v = FIRST ? a.uvel[i] : a.vel0[i];
            ax = FIRST ? aux_pack(a.urad[i], a.utype[i], i) : a.aux0[i];
        }
    }
    for (int j = tid; j < a.n; j += kFlatThreads) {
        const float2 c = pos[j];
        keys[j] = x_order_key(by_y ? c.y : c.x);
    }
    if (FIRST && q == 0 && i < a.n &&
        !(isfinite(p.x) && isfinite(p.y) && isfinite(v.x) && isfinite(v.y)))
        atomicOr(a.err, ERR_BIT_NONFINITE);
    __syncthreads();
    const uint32_t own = x_order_key(by_y ? p.y : p.x);
    uint32_t rank = 0u;
#pragma unroll 4
    for (int j = q; j < a.n; j += kFlatLanes) {
        const uint32_t k = keys[j];
        rank += (k < own || (k == own && j < i)) ? 1u : 0u;
    }
#pragma unroll
    for (int d = 1; d < kFlatLanes; d <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, d);
    if (q == 0 && i < a.n) {
        a.pos1[rank] = p;
        a.vel1[rank] = v;
        a.aux1[rank] = ax;
    }
}

}  // namespace orca
