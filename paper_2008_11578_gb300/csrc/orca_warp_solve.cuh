// orca_warp_solve.cuh -- the solve kernel with one warp per agent (sm_103a).
//
// For scenes too small to fill the GPU with one thread per agent, where the
// step waits for one thread's serial chain (search, k half-planes, LP) and
// most SMs idle.  The warp's 32 lanes split each part of that chain:
//   search       32 candidates per load; the list is one entry per lane
//   half-planes  one per lane
//   LP           a sub-problem's bounds one per lane, merged by redux; the
//                next violated line is found by a vote, not by a loop
// Every expression and every discrete choice is the per-thread kernel's
// (agent_solve_kernel), so a step's results do not depend on which one ran.
// Bound by the latency of one agent's chain while the scene is small (4,000
// agents: 49 -> 17 us a launch; with cells, as in a batch, 1,000 agents take 14 us,
// about 12,500 cycles an agent: loads 1,600, seed 2,100, scan 1,900, half-planes
// 1,400, order 900, LP 3,600), then by issue slots (16,000 agents: 51 -> 40 us,
// 73 % of issue slots busy; eight blocks an SM 39.7 us, seven 40.9, six 41.0,
// five 43.0).
#pragma once

#include "orca_step_kernels.cuh"

namespace orca {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMergeMin = 6;   // candidates from which one merge beats single insertions

__device__ __forceinline__ float redux_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float redux_min(float x) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ unsigned long long shfl64(unsigned long long x, int src) {
    return __shfl_sync(kFull, x, src);
}

// Per-warp shared memory: the lines in LP order; the search's keys (the
// candidates' and the list's d^2) and its lanes by rank.
struct WarpSlots {
    float4 line[32];
    float d2[32];
    float list[32];
    int lane[32];
};

// How many of the 32 values are below x.
__device__ __forceinline__ int count_below(const float* v, float x) {
    int r = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 e = *reinterpret_cast<const float4*>(v + 4 * u);
        r += (e.x < x ? 1 : 0) + (e.y < x ? 1 : 0) + (e.z < x ? 1 : 0) + (e.w < x ? 1 : 0);
    }
    return r;
}

// Interval of a 1D sub-problem after the bounds of the lanes that have one
// (upper: t <= tt, lower: t >= tt) are merged into [tl, tr]; with ACT, kl and kr
// name the first lane that set each end (-1: none did).  A lane that finds the
// sub-problem empty (empty) puts the lower end at infinity.
template <bool ACT>
__device__ __forceinline__ void merge_bounds(bool upper, bool lower, bool empty, float tt,
                                             float& tl, float& tr, int& kl, int& kr) {
    const float hi = redux_min(upper ? tt : CUDART_INF_F);
    const float lo = redux_max(empty ? CUDART_INF_F : (lower ? tt : -CUDART_INF_F));
    if (ACT) {
        const unsigned mr = __ballot_sync(kFull, upper && tt == hi);
        const unsigned ml = __ballot_sync(kFull, lower && tt == lo);
        kr = hi < tr ? __ffs(mr) - 1 : -1;
        kl = lo > tl ? __ffs(ml) - 1 : -1;
    }
    tr = fminf(tr, hi);
    tl = fmaxf(tl, lo);
}

// lp2_project over the warp: lane j holds line lj (j < n), L the same lines.
template <bool ACT>
__device__ __forceinline__ int warp_lp2(const float4* L, float4 lj, int lane, int n, float vmax,
                                        float vpx, float vpy, float& vx, float& vy,
                                        uint32_t& act) {
    const float tol = lp_tol(vmax);
    const bool capped = disc_project(vmax, vpx, vpy, vx, vy);
    act = act_pack(ACT_PROJ, capped, 0, 0, 0, 0);
    int done = -1;   // lines up to this one are satisfied
    for (;;) {
        const unsigned m = __ballot_sync(
            kFull, lane < n && lane > done && penetration(lj, vx, vy) > 0.0f);
        if (m == 0u) return n;
        const int i = __ffs(m) - 1;
        done = i;
        const float4 li = L[i];
        float tl, tr;
        if (!disc_chord(li.x, li.y, li.z, li.w, vmax, tol, tl, tr)) return i;
        float den, num;
        line_bound(li, lj, den, num);
        const bool on = lane < i;
        const float tt = __fdividef(num, den);
        int kl = -1, kr = -1;
        merge_bounds<ACT>(on && den > 0.0f, on && den < 0.0f, on && den == 0.0f && num < -tol, tt,
                          tl, tr, kl, kr);
        if (tl > tr + tol) return i;
        const float t0 = line_project(li, vpx, vpy, tl, tr, vx, vy);
        const int bound = (t0 > tr) ? kr : ((t0 < tl) ? kl : -2);
        act = bound >= 0 ? act_pack(ACT_PROJ, false, 2, i, bound, 0)
                         : act_pack(ACT_PROJ, bound == -1, 1, i, 0, 0);
    }
}

// lp3_min_penetration over the warp.
template <bool ACT>
__device__ __forceinline__ float warp_lp3(const float4* L, float4 lj, int lane, int n, float vmax,
                                          float sx, float sy, float& vx, float& vy, uint32_t& act,
                                          bool& fallback) {
    const float tol = lp_tol(vmax);
    const float cj = penetration(lj, sx, sy);   // det(d, P - s)
    const float4 l0 = L[0];
    vx = __fmul_rn(-l0.w, vmax);
    vy = __fmul_rn(l0.z, vmax);
    act = act_pack(ACT_VERTEX, true, 1, 0, 0, 0);
    float t = penetration(l0, vx, vy);
    int done = 0;
    for (;;) {
        const unsigned m = __ballot_sync(
            kFull, lane < n && lane > done && !(penetration(lj, vx, vy) <= t));
        if (m == 0u) break;
        const int i = __ffs(m) - 1;
        done = i;
        const float4 li = L[i];
        const float nix = -li.w, niy = li.z;   // objective: maximise n_i . v
        float cx = __fmul_rn(vmax, nix), cy = __fmul_rn(vmax, niy);
        uint32_t ai = act_pack(ACT_VERTEX, true, 1, i, 0, 0);
        // every lane's plane against plane i
        const PlanePair q = plane_pair(li, __shfl_sync(kFull, cj, i), lj, cj);
        int seen = -1;
        for (;;) {
            const unsigned mj = __ballot_sync(
                kFull, lane < i && lane > seen && plane_above(q, cx, cy, sx, sy));
            if (mj == 0u) break;
            const int j = __ffs(mj) - 1;
            seen = j;
            PlanePair qj;
            qj.ax = __shfl_sync(kFull, q.ax, j);
            qj.ay = __shfl_sync(kFull, q.ay, j);
            qj.a2 = __shfl_sync(kFull, q.a2, j);
            qj.beta = __shfl_sync(kFull, q.beta, j);
            if (qj.a2 <= 1e-12f) continue;   // same direction: one plane dominates
            const PairLine b = pair_line(qj, sx, sy);
            float tl, tr;
            if (!disc_chord(b.bx, b.by, b.ex, b.ey, vmax, tol, tl, tr)) {
                fallback = true;
                continue;
            }
            float den, num;
            pair_bound(q, b, den, num);
            const bool on = lane < j && !(q.a2 <= 1e-12f);
            const float tt = __fdividef(num, den);
            int kl = -1, kr = -1;
            merge_bounds<ACT>(on && den < 0.0f, on && den > 0.0f, on && den == 0.0f && num > tol,
                              tt, tl, tr, kl, kr);
            if (tl > tr + tol) {   // empty only through rounding: keep the point
                fallback = true;
                continue;
            }
            const bool right = mul_add(nix, b.ex, niy, b.ey) > 0.0f;
            const float te = right ? tr : tl;
            const int kb = right ? kr : kl;
            cx = __fmaf_rn(te, b.ex, b.bx);
            cy = __fmaf_rn(te, b.ey, b.by);
            ai = kb >= 0 ? act_pack(ACT_VERTEX, false, 3, i, j, kb)
                         : act_pack(ACT_VERTEX, true, 2, i, j, 0);
        }
        vx = cx;
        vy = cy;
        act = ai;
        t = penetration(li, vx, vy);
    }
    return redux_max(lane < n ? penetration(lj, vx, vy) : -CUDART_INF_F);
}

// solve_velocity over the warp.
template <bool ACT>
__device__ __forceinline__ int warp_solve_velocity(const float4* L, float4 lj, int lane, int n,
                                                   float vmax, float vpx, float vpy, float sx,
                                                   float sy, float& vx, float& vy, float& tstar,
                                                   uint32_t& act) {
    tstar = 0.0f;
    float v3x = 0.0f, v3y = 0.0f, t3 = -CUDART_INF_F;
    uint32_t act3 = 0u;
    bool fallback = false;
    if (n > 0) t3 = warp_lp3<ACT>(L, lj, lane, n, vmax, sx, sy, v3x, v3y, act3, fallback);
    if ((t3 <= 0.1f * lp_tol(vmax) || fallback || n == 0) &&
        warp_lp2<ACT>(L, lj, lane, n, vmax, vpx, vpy, vx, vy, act) == n)
        return 0;
    act = act3;
    tstar = t3;
    vx = v3x;
    vy = v3y;
    // valley: the first exactly opposite pair, in index order, of the lines
    // that attain t*
    const unsigned am = __ballot_sync(
        kFull, lane < n && !(penetration(lj, v3x, v3y) < attains_limit(t3)));
    int vi = -1, vj = -1;
    for (unsigned m = am; m != 0u; m &= m - 1u) {
        const int i = __ffs(m) - 1;
        const unsigned mo = __ballot_sync(
            kFull, lane > i && ((am >> lane) & 1u) && opposite(L[i], lj));
        if (mo != 0u) {
            vi = i;
            vj = __ffs(mo) - 1;
            break;
        }
    }
    if (vi >= 0) {
        float ox, oy;
        int work = 0;
        if (valley_project(L, 1, n, vi, vj, t3, vmax, vpx, vpy, ox, oy, work, act)) {
            vx = ox;
            vy = oy;
        }
    }
    return 1;
}

// The new state of agent o at slot s: integration, output, binning for the next step.
__device__ __forceinline__ void write_step(const SceneDev& sc, int s, int o, float2 p, float2 v,
                                           float2 vn, const StepOut& out, const DebugOut& dbg) {
    const float2 pn = make_float2(__fadd_rn(p.x, __fmul_rn(sc.dt, vn.x)),
                                  __fadd_rn(p.y, __fmul_rn(sc.dt, vn.y)));
    const int w = out.caller_order ? o : s;
    out.vel[w] = vn;
    out.pos[w] = pn;
    if (out.hint != nullptr) {
        out.hint[s] = (uint32_t)o;
        if (s == 0) *out.hint_ok = 1;
    }
    if (out.key != nullptr) {
        const int ncx = cell_axis(pn.x, sc.origin_x, sc.inv_cell_x, sc.nx);
        const int ncy = cell_axis(pn.y, sc.origin_y, sc.inv_cell_y, sc.ny);
        const uint32_t c = (uint32_t)(sc.cell_off + ncy * sc.nx + ncx);
        out.key[s] = c;
        out.slot[s] = atomicAdd(out.count + c, 1u);
    }
    if (dbg.spos != nullptr) dbg.spos[o] = p;
    if (dbg.svel != nullptr) dbg.svel[o] = v;
    if (dbg.vnew != nullptr) dbg.vnew[o] = vn;
}

// The rest of an agent's step by one lane, in the sorted-list kernel's order of
// lines and of operations, for half-planes that are no numbers or beyond all
// measure: there a vote, a minimum over the lanes and a loop over the lines differ
// in what they make of an overflow.  W.line holds the n lines in neighbour order.
// (Out of line and to the end of the step: what comes back into the kernel from
// here costs its registers 4 to 11 % of the time of 16,000 agents; like this 1.5 %.)
template <bool ACT>
__device__ __noinline__ void finish_by_one_lane(WarpSlots& W, int n, float vmax, float2 vp, float2 p,
                                                float2 v, int s, int o, int cnt, bool any_overlap,
                                                unsigned capbits, unsigned ovbits, SceneDev sc,
                                                StepOut out, DebugOut dbg) {
    float4* line = W.line;
    int* order = W.lane;
    auto pen = [&](int i) { return penetration(line[i], v.x, v.y); };
    auto swap = [&](int a, int b) {
        const float4 l = line[a];
        line[a] = line[b];
        line[b] = l;
        const int t = order[a];
        order[a] = order[b];
        order[b] = t;
    };
    float pm0 = -CUDART_INF_F, pm1 = -CUDART_INF_F;
    int im0 = -1, im1 = -1;
    for (int i = 0; i < n; ++i) {
        order[i] = i;
        const float pv = pen(i);
        if (pv > pm0) {
            pm1 = pm0;
            im1 = im0;
            pm0 = pv;
            im0 = i;
        } else if (pv > pm1) {
            pm1 = pv;
            im1 = i;
        }
    }
    if (im0 > 0) swap(0, im0);
    if (im1 >= 0 && n > 2) {
        const int b = im1 == 0 ? im0 : im1;
        if (b > 1) swap(1, b);
    }
    if (n <= 16)
        for (int m = 3; m < n; ++m)
            for (int at = m; at > 2 && pen(at - 1) < pen(at); --at) swap(at - 1, at);
    float vx, vy, tstar;
    uint32_t act = 0u;
    int work = 0;
    const int infeasible = solve_velocity(
        line, 1, n, vmax, vp.x, vp.y, v.x, v.y,
        [&](int, float4 l) { return penetration(l, v.x, v.y); }, vx, vy, tstar, work, act);
    if (ACT && dbg.act != nullptr) {
        const int nl = act_nlines(act);
        for (int m = 0; m < nl; ++m) {
            const int li = order[act_line(act, m)];
            act = (act & ~(31u << (8 + 8 * m))) | ((uint32_t)li << (8 + 8 * m));
            act |= ((capbits >> li) & 1u) << (13 + 8 * m);
            act |= ((ovbits >> li) & 1u) << (14 + 8 * m);
        }
        dbg.act[o] = act;
    }
    write_step(sc, s, o, p, v, make_float2(vx, vy), out, dbg);
    if (dbg.cell != nullptr)
        dbg.cell[o] = cell_axis(p.y, sc.origin_y, sc.inv_cell_y, sc.ny) * sc.nx +
                      cell_axis(p.x, sc.origin_x, sc.inv_cell_x, sc.nx);
    if (dbg.cnt != nullptr) dbg.cnt[o] = cnt;
    if (dbg.flags != nullptr) dbg.flags[o] = (uint8_t)(infeasible | (any_overlap ? 4 : 0));
    if (dbg.tstar != nullptr) dbg.tstar[o] = tstar;
}

// One warp per agent (sorted slot s).  MODE_PLAIN or MODE_RECORD, the
// incremental LP, and at most 32 lines (k plus the vehicles' kinematic ones).
//
// Search: the seed takes one candidate per lane from the agent's row and the
// rows around it and ranks them by (d^2, index) in one pass; the k-th of them
// bounds what is left.  Rows whose seed did not reach that bound on a side, and then
// the rows farther out, are scanned in chunks of 16 slots each way; a
// candidate below the bound enters the list (one entry per lane, sorted) by
// one shift of the lanes behind it.  The list is the set of the k smallest
// keys whatever the order of the candidates, so it equals the per-thread
// kernel's.
//
// FLAT: the smallest scenes, not binned into cells but sorted by one coordinate
// (y if by_y, else x): one row of all slots, 16 on either side of the agent
// seed the list, and both sides go on until the coordinate alone is beyond the
// bound; the first 32 slots after the seed's are loaded with it, each later 32
// while the ones before are tested.
template <class SRC, int MODE, bool FLAT>
__global__ void __launch_bounds__(128, 8)
warp_solve_kernel(int n, bool by_y, SRC src, const float2* pos, const float2* vel,
                  const uint2* aux, const uint32_t* cstart, AgentIn ain,
                  const float2* __restrict__ vpd, StepOut out, DebugOut dbg,
                  int* __restrict__ err) {
    __shared__ WarpSlots slots[4];
    const int lane = threadIdx.x & 31;
    WarpSlots& W = slots[threadIdx.x >> 5];
    const int s = lane_group(blockIdx.x, blockDim.x, threadIdx.x, 32u);
    launch_dependents();
    wait_for_primary();
    if (s >= n) return;
    const SceneDev& sc = src.get(s);
    const int status = __ldcg(err);
    const float2 p = pos[s];
    const float2 v = vel[s];
    const uint2 as = aux[s];
    // no index read from the sorted state is followed before this
    if (status & (ERR_BIT_TIMEOUT | ERR_BIT_STATE)) return;
    const float r = aux_rad(as);
    const int ta = aux_type(as);
    const int o = aux_orig(as);
    const int cx = cell_axis(p.x, sc.origin_x, sc.inv_cell_x, sc.nx);
    const int cy = cell_axis(p.y, sc.origin_y, sc.inv_cell_y, sc.ny);
    const int k = sc.k;

    // ---- target (its loads overlap the search's) ----
    float2 g = ain.goal[o];
    const float vmax = ain.max_speed[o];
    const float2 offset = vpd != nullptr ? vpd[o] : make_float2(0.0f, 0.0f);
    if (ain.route != nullptr) {
        const int rt = ain.route[o];
        if (rt >= 0) {
            int wi = ain.wp_idx[o];
            if (lane == 0 && dbg.swp != nullptr) dbg.swp[o] = (uint8_t)wi;
            wi = advance_waypoint(ain.waypoints + (size_t)rt * ain.n_waypoints, ain.n_waypoints,
                                  wi, p, r, g);
            __syncwarp();   // every lane has read the index
            if (lane == 0) {
                ain.wp_idx[o] = (uint8_t)wi;
                if (dbg.wp_used != nullptr) dbg.wp_used[o] = (uint8_t)wi;
            }
        }
    }

    // ---- k nearest by (d^2, index) ----
    // lane m < cnt: the m-th nearest, its key and sorted slot
    unsigned long long key = ~0ull;
    int slot = -1, cnt = 0;
    if (k > 0 && isfinite(p.x) && isfinite(p.y)) {
        const float R2 = sc.R2;
        const float thr0 = R2 > 0.0f ? __int_as_float(__float_as_int(R2) - 1) : -1.0f;
        const uint32_t* cs = cstart + sc.cell_off;
        const int nx = sc.nx, ny = sc.ny;
        const float ch = sc.cell_h, mg = sc.ring_delta * ch;
        const float pry = __fsub_rn(p.y, sc.origin_y);
        auto row_gap2 = [&](int ry) {
            const float by0 = ry == 0 ? -CUDART_INF_F : (float)ry * ch - mg;
            const float by1 = ry == ny - 1 ? CUDART_INF_F : (float)(ry + 1) * ch + mg;
            const float ey = fmaxf(fmaxf(by0 - pry, pry - by1), 0.0f);
            return ey * ey * 0.99999f;
        };
        const float fx = fminf(fmaxf(__fmul_rn(__fsub_rn(p.x, sc.origin_x), sc.inv_cell_x) -
                                         (float)cx, 0.0f), 1.0f);
        // slot ranges of the rows row0 .. row0 + 7, loaded at once: lane
        // 4 i + q holds row row0 + i's begin, end, and the begin and end of
        // its cell of column cx
        int row0 = cy - 3;
        int range = 0;
        auto load_rows = [&]() {
            const int ry = row0 + (lane >> 2), q = lane & 3;
            range = 0;
            if (ry >= 0 && ry < ny)
                range = (int)cs[(size_t)ry * nx + (q == 0 ? 0 : q == 1 ? nx : cx + q - 2)];
        };
        if (!FLAT) load_rows();
        // ---- seed ----
        bool sparse = false, left = lane >= 16;
        int off = 0, step = lane & 15, half = 16;   // row offset, place in the row's lanes
        int rb = 0, re = n, start = s;
        float g2s = 0.0f;
        float2 ahead[2];          // FLAT: the slots after the seed's, rightward and leftward
        uint32_t ahead_idx[2];
        auto load = [&](int j, float2& c, uint32_t& oc) {
            if (j >= 0 && j < n) {
                c = pos[j];
                oc = aux[j].y;
            }
        };
        if (FLAT) {
            load(s + 17 + lane, ahead[0], ahead_idx[0]);
            load(s - 17 - lane, ahead[1], ahead_idx[1]);
        } else {
            step = lane & 7;
            half = 4;
            // Lanes 0-7 take the own row; the others the rows around it, nearest
            // slots first, half of them each way.  Dense: 8 each way in the own
            // row and 4 in the rows next to it.  Sparse (the k-th neighbour is
            // probably beyond the next row, judged by the agents in the own
            // column's three cells): 4 in the own row, 3 in two rows on each side.
            const int i0 = (cy - row0) << 2;
            int column = __shfl_sync(kFull, range, i0 + 3) - __shfl_sync(kFull, range, i0 + 2);
            column += __shfl_sync(kFull, range, i0 - 1) - __shfl_sync(kFull, range, i0 - 2);
            column += __shfl_sync(kFull, range, i0 + 7) - __shfl_sync(kFull, range, i0 + 6);
            sparse = 3.0f * (float)k * sc.cell_w > 4.5f * (float)column * ch;
            if (sparse) {
                if (lane >= 8) {
                    const int u = lane - 8;   // 6 lanes for each of rows -1, +1, -2, +2
                    const int w = u / 6;
                    off = (w & 1 ? 1 : -1) * (1 + (w >> 1));
                    step = u - 6 * w;
                    half = 3;
                }
            } else if (lane < 16) {
                step = lane;
                half = 8;
            } else {
                off = lane < 24 ? -1 : 1;
            }
            left = step >= half;
            if (left) step -= half;
            const int ib = i0 + 4 * off;
            rb = __shfl_sync(kFull, range, ib);
            re = __shfl_sync(kFull, range, ib + 1);
            const int bc = __shfl_sync(kFull, range, ib + 2), ec = __shfl_sync(kFull, range, ib + 3);
            start = off == 0 ? s : min(bc + (int)(fx * (float)(ec - bc)), ec);
            g2s = off == 0 ? 0.0f : row_gap2(cy + off);
        }
        const int js = left ? start - 1 - step : start + (off == 0 ? 1 : 0) + step;
        const bool in = js >= rb && js < re;
        // distance along the rows (dx, or dy when sorted by y), its square, d^2
        auto measure = [&](float2 c, float& along, float& along2) {
            const float dx = __fsub_rn(c.x, p.x), dy = __fsub_rn(c.y, p.y);
            const float xx = __fmul_rn(dx, dx), yy = __fmul_rn(dy, dy);
            along = FLAT && by_y ? dy : dx;
            along2 = FLAT && by_y ? yy : xx;
            return __fadd_rn(xx, yy);
        };
        float ds = CUDART_INF_F, dxs = 0.0f, dxxs = 0.0f;
        uint32_t os = 0u;
        if (in) {
            os = aux[js].y;
            const float d2 = measure(pos[js], dxs, dxxs);
            if (d2 <= thr0) ds = d2;
        }
        const int oj = aux_orig(make_uint2(0u, os));
        const bool pass = ds < CUDART_INF_F;
        const unsigned pm = __ballot_sync(kFull, pass);
        W.d2[lane] = ds;
        __syncwarp();
        // rank by d^2; lanes that share a rank (equal d^2) are told apart by index
        int rank = count_below(W.d2, ds);
        if (pass) W.lane[rank] = lane;
        __syncwarp();
        if (__any_sync(kFull, pass && W.lane[rank] != lane)) {
            __syncwarp();
            unsigned same = __match_any_sync(kFull, __float_as_uint(ds)) & ~(1u << lane);
            if (!pass) same = 0u;
            while (__any_sync(kFull, same != 0u)) {
                const int ou = __shfl_sync(kFull, oj, same != 0u ? __ffs((int)same) - 1 : lane);
                if (same != 0u && ou < oj) ++rank;
                same &= same - 1u;
            }
            if (pass) W.lane[rank] = lane;
            __syncwarp();
        }
        cnt = min(__popc(pm), k);
        {
            const int from = lane < cnt ? W.lane[lane] : 0;
            const float d = __shfl_sync(kFull, ds, from);
            const int of = __shfl_sync(kFull, oj, from);
            const int jf = __shfl_sync(kFull, js, from);
            if (lane < cnt) {
                key = ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)of;
                slot = jf;
            }
        }
        float thr_d = thr0;   // as in the per-thread search
        auto update = [&]() {
            if (cnt == k)
                thr_d = __uint_as_float(__shfl_sync(kFull, (unsigned)(key >> 32), k - 1));
        };
        update();
        // candidates ck (slots j) of the lanes in am enter the list: one by one,
        // each shifting the entries behind it, or, when there are many, all at
        // once by their ranks in the merged list (unless equal d^2 have to be
        // told apart by index)
        auto admit = [&](unsigned am, unsigned long long ck, int j) {
            const int c = __popc(am);
            if (c >= kMergeMin) {
                const bool cand = (am >> lane) & 1u, held = lane < cnt;
                const float cd = cand ? __uint_as_float((unsigned)(ck >> 32)) : CUDART_INF_F;
                const float ld = held ? __uint_as_float((unsigned)(key >> 32)) : CUDART_INF_F;
                __syncwarp();
                W.d2[lane] = cd;
                W.list[lane] = ld;
                __syncwarp();
                const int rc = count_below(W.d2, cd) + count_below(W.list, cd);
                const int rl = lane + count_below(W.d2, ld);
                if (held && rl < 32) W.lane[rl] = lane;
                if (cand && rc < 32) W.lane[rc] = 32 + lane;
                __syncwarp();
                const bool tie = (held && rl < 32 && W.lane[rl] != lane) ||
                                 (cand && rc < 32 && W.lane[rc] != 32 + lane);
                if (!__any_sync(kFull, tie)) {
                    cnt = min(cnt + c, k);
                    const int from = lane < cnt ? W.lane[lane] : 0;
                    const unsigned long long a = shfl64(key, from & 31), b = shfl64(ck, from & 31);
                    const int ja = __shfl_sync(kFull, slot, from & 31);
                    const int jb = __shfl_sync(kFull, j, from & 31);
                    key = lane < cnt ? (from < 32 ? a : b) : ~0ull;
                    slot = from < 32 ? ja : jb;
                    update();
                    return;
                }
            }
            while (am != 0u) {
                const int from = __ffs(am) - 1;
                am &= am - 1u;
                const unsigned long long x = shfl64(ck, from);
                const int xj = __shfl_sync(kFull, j, from);
                const unsigned long long up = __shfl_up_sync(kFull, key, 1);
                const int uj = __shfl_up_sync(kFull, slot, 1);
                const bool below = x < key;   // entries behind the candidate shift
                const bool shift = lane > 0 && x < up;
                if (below) {
                    key = shift ? up : x;
                    slot = shift ? uj : xj;
                }
            }
            cnt = min(cnt + c, k);
            if (lane >= k) key = ~0ull;   // pushed out of the list
            update();
        };
        // candidate c (index word oc) at slot j of a row whose y gap^2 is g2:
        // enters the list when below the bound; returns whether it and all
        // farther ones on its side are beyond it
        auto test_loaded = [&](bool on, int j, bool lf, float g2, float2 c, uint32_t oc) {
            float d2 = CUDART_INF_F, dx = 0.0f, dxx = 0.0f;
            if (on) d2 = measure(c, dx, dxx);
            const bool cand = on && d2 <= thr_d;
            if (__ballot_sync(kFull, cand) != 0u) {
                // (of many at the k-th's distance only those with a smaller index:
                // 16,000 agents at 16 points 729 -> 211 us a step)
                const unsigned long long ck = ((unsigned long long)__float_as_uint(d2) << 32) |
                                              (unsigned)aux_orig(make_uint2(0u, oc));
                const unsigned long long last = shfl64(key, k - 1);   // (every lane takes part)
                const unsigned am = __ballot_sync(kFull, cand && ck < last);
                if (am != 0u) admit(am, ck, j);
            }
            return !on || ((lf ? dx < 0.0f : dx > 0.0f) && __fadd_rn(dxx, g2) > thr_d);
        };
        auto test = [&](bool on, int j, bool lf, float g2) {
            float2 c = make_float2(0.0f, 0.0f);
            uint32_t oc = 0u;
            if (on) load(j, c, oc);
            return test_loaded(on, j, lf, g2, c, oc);
        };
        // The seeded rows go on from where their seed ended, 32 slots at a time,
        // on the sides that it left open: a side is finished when a candidate on
        // it is beyond the bound (all farther ones are) or when the row ends.
        const unsigned fin = __ballot_sync(
            kFull, !in || ((left ? dxs < 0.0f : dxs > 0.0f) && __fadd_rn(dxxs, g2s) > thr_d));
        const unsigned my_side = ((1u << half) - 1u) << (lane - step);
        unsigned open = __ballot_sync(kFull,
                                      step == 0 && (fin & my_side) == 0u && g2s <= thr_d);
        if (FLAT) {
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const bool lf = side == 1;
                if ((open & (lf ? 0xffff0000u : 0xffffu)) == 0u) continue;
                int j = lf ? s - 17 - lane : s + 17 + lane;
                for (;;) {
                    const float2 c = ahead[side];
                    const uint32_t oc = ahead_idx[side];
                    const int next = lf ? j - 32 : j + 32;
                    load(next, ahead[side], ahead_idx[side]);
                    if (__ballot_sync(kFull, test_loaded(j >= 0 && j < n, j, lf, 0.0f, c, oc)) !=
                        0u)
                        break;
                    j = next;
                }
            }
            open = 0u;
        }
        for (; open != 0u; open &= open - 1u) {
            const int u = __ffs(open) - 1;   // the side's first lane
            const bool lf = __shfl_sync(kFull, left ? 1 : 0, u) != 0;
            const int b = __shfl_sync(kFull, rb, u), e = __shfl_sync(kFull, re, u);
            const float g2 = __shfl_sync(kFull, g2s, u);
            int j = __shfl_sync(kFull, js, u);
            const int h = __shfl_sync(kFull, half, u);
            j += lf ? -h - lane : h + lane;
            while (__ballot_sync(kFull, test(j >= b && j < e, j, lf, g2)) == 0u)
                j += lf ? -32 : 32;
        }
        // The rows farther out, 16 slots each way at a time; a side ends at the
        // grid edge or at the first row whose y gap is beyond the bound.
        bool up = !FLAT, down = !FLAT;
        for (int m = sparse ? 3 : 2; up || down; ++m) {
            const float gd = row_gap2(cy - m), gu = row_gap2(cy + m);
            const int first = gu < gd ? 1 : 0;
            for (int so = 0; so < 2; ++so) {
                const int side = so ^ first;
                if (!(side == 0 ? down : up)) continue;
                const int ry = side == 0 ? cy - m : cy + m;
                const float g2 = side == 0 ? gd : gu;
                if (ry < 0 || ry >= ny || g2 > thr_d) {
                    if (side == 0) down = false;
                    else up = false;
                    continue;
                }
                if (ry < row0 || ry > row0 + 7) {
                    row0 = side == 0 ? ry - 7 : ry;
                    load_rows();
                }
                const int i = (ry - row0) << 2;
                const int b = __shfl_sync(kFull, range, i), e = __shfl_sync(kFull, range, i + 1);
                const int bc = __shfl_sync(kFull, range, i + 2);
                const int ec = __shfl_sync(kFull, range, i + 3);
                const int at = min(bc + (int)(fx * (float)(ec - bc)), ec);
                const bool lf = lane >= 16;
                int j = lf ? at - 1 - (lane - 16) : at + lane;
                bool ron = true, lon = true;
                while (ron || lon) {
                    const unsigned sm = __ballot_sync(
                        kFull, test((lf ? lon : ron) && j >= b && j < e, j, lf, g2));
                    ron = ron && (sm & 0xffffu) == 0u;
                    lon = lon && (sm >> 16) == 0u;
                    j += lf ? -16 : 16;
                }
            }
        }
    }
    const bool mine = lane < cnt;
    const int onbr = (int)(unsigned)(key & 0xffffffffull);
    if (dbg.nbr != nullptr && lane < dbg.k_stride)
        dbg.nbr[(size_t)o * dbg.k_stride + lane] = mine ? onbr : -1;

    // ---- one ORCA half-plane per lane, then the vehicles' kinematic ones ----
    float4 line = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    bool cap = false, ov = false;
    if (mine) {
        const float2 pj = pos[slot], vj = vel[slot];
        const uint2 aj = aux[slot];
        const float rj = aux_rad(aj);
        const int tb = aux_type(aj);
        const float rs = __fadd_rn(r, rj);
        ov = __uint_as_float((unsigned)(key >> 32)) <= __fmul_rn(rs, rs);
        const float f = tb ? (ta ? sc.f11 : sc.f01) : (ta ? sc.f10 : sc.f00);
        line = orca_line(p.x, p.y, v.x, v.y, r, pj.x, pj.y, vj.x, vj.y, rj, f, sc.inv_tau,
                         sc.inv_dt, ov, cap);
    }
    const bool any_overlap = __any_sync(kFull, ov);
    const float2 vp = preferred_velocity(p, g, vmax, sc.inv_dt, vpd != nullptr, offset);
    int nlines = cnt;
    if (ta != 0 && (sc.kin_turn || sc.kin_accel))
        limit_lines(sc, v, vp, [&](float4 l) {
            if (lane == nlines) line = l;
            ++nlines;
        });

    // (beyond these sizes the LP's products overflow)
    const float size = (lane < nlines ? fabsf(line.x) + fabsf(line.y) : 0.0f) + fabsf(v.x) +
                       fabsf(v.y) + vmax;
    if (__any_sync(kFull, !(size < 1e12f) || vmax < 0.0f)) {
        const unsigned capbits = __ballot_sync(kFull, cap), ovbits = __ballot_sync(kFull, ov);
        __syncwarp();
        if (lane < nlines) W.line[lane] = line;
        __syncwarp();
        if (lane == 0)
            finish_by_one_lane<MODE == MODE_RECORD>(W, nlines, vmax, vp, p, v, s, o, cnt,
                                                    any_overlap, capbits, ovbits, sc, out, dbg);
        return;
    }

    // ---- constraint order of the LP (the per-thread kernel's) ----
    // The two lines most violated at v_A swap into slots 0 and 1; with at
    // most 16 lines the others follow by decreasing penetration, equal ones
    // in the order those swaps leave.
    int place = lane;
    if (nlines > 1) {
        float pv = lane < nlines ? penetration(line, v.x, v.y) : -CUDART_INF_F;
        if (!(pv == pv)) pv = -CUDART_INF_F;
        const float p0 = redux_max(pv);
        const unsigned m0 = __ballot_sync(kFull, pv == p0 && pv > -CUDART_INF_F);
        const int im0 = __ffs(m0) - 1;
        const float pw = lane == im0 ? -CUDART_INF_F : pv;
        const float p1 = redux_max(pw);
        const unsigned m1 = __ballot_sync(kFull, pw == p1 && pw > -CUDART_INF_F);
        const int im1 = __ffs(m1) - 1;
        if (im0 > 0) place = lane == im0 ? 0 : (lane == 0 ? im0 : lane);
        if (im1 >= 0 && nlines > 2) {
            const int b = im1 == 0 ? im0 : im1;   // where the second line is now (>= 1)
            if (b > 1) place = place == b ? 1 : (place == 1 ? b : place);
        }
        if (nlines <= 16 && nlines > 3) {
            if (lane < 16) W.d2[lane < nlines ? place : lane] = pv;   // -inf beyond the lines
            __syncwarp();
            int before = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 e = *reinterpret_cast<const float4*>(&W.d2[4 * u]);
                const int at = 4 * u;
                if (u > 0) {
                    before += (e.x > pv || (e.x == pv && at < place)) ? 1 : 0;
                    before += (e.y > pv || (e.y == pv && at + 1 < place)) ? 1 : 0;
                }
                before += (e.z > pv || (e.z == pv && at + 2 < place)) ? 1 : 0;
                before += (e.w > pv || (e.w == pv && at + 3 < place)) ? 1 : 0;
            }
            if (lane < nlines && place >= 2) place = 2 + before;
        }
    }
    __syncwarp();   // the seed's use of the slots is over
    if (lane < nlines) W.line[place] = line;
    if (MODE == MODE_RECORD) W.lane[place] = lane;   // lanes beyond the lines keep their own place
    __syncwarp();
    const float4 lj = W.line[lane < nlines ? lane : 0];

    // ---- velocity LP, least-penetration fallback ----
    float vx, vy, tstar;
    uint32_t act = 0u;
    const int infeasible = warp_solve_velocity<MODE == MODE_RECORD>(
        W.line, lj, lane, nlines, vmax, vp.x, vp.y, v.x, v.y, vx, vy, tstar, act);
    if (MODE == MODE_RECORD && dbg.act != nullptr) {
        // line indices back in neighbour order, with each line's construction
        const unsigned capbits = __ballot_sync(kFull, cap), ovbits = __ballot_sync(kFull, ov);
        const int nl = act_nlines(act);
        for (int m = 0; m < nl; ++m) {
            const int li = W.lane[act_line(act, m)];
            act = (act & ~(31u << (8 + 8 * m))) | ((uint32_t)li << (8 + 8 * m));
            act |= ((capbits >> li) & 1u) << (13 + 8 * m);
            act |= ((ovbits >> li) & 1u) << (14 + 8 * m);
        }
    }

    // ---- integrate ----
    if (lane != 0) return;
    write_step(sc, s, o, p, v, make_float2(vx, vy), out, dbg);
    if (MODE == MODE_RECORD && dbg.act != nullptr) dbg.act[o] = act;
    if (dbg.cell != nullptr) dbg.cell[o] = cy * sc.nx + cx;
    if (dbg.cnt != nullptr) dbg.cnt[o] = cnt;
    if (dbg.flags != nullptr) dbg.flags[o] = (uint8_t)(infeasible | (any_overlap ? 4 : 0));
    if (dbg.tstar != nullptr) dbg.tstar[o] = tstar;
}

}  // namespace orca
