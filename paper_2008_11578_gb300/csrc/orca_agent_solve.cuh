// orca_agent_solve.cuh -- the solve kernel with one thread per agent (sm_103a).
//
// Search: the k + 1 smallest distances are kept sorted in registers by a
// network of minima and maxima (no branches: the 32 lanes of a warp insert
// whatever their candidates are).  An entry is the distance d^2 with its lowest
// bits replaced by the candidate's place in a list of admitted slots in shared
// memory, so the order of the neighbours falls out of the network.  Where two
// distances differ only in the replaced bits (some 5e-4 of the agents, or every
// one on a regular grid) the run of them is put in order exactly (order_ties):
// 1M agents on a grid of 1 m 392 -> 238 us against an ordering of the whole list by
// all pairs (186 with a sorted list in shared memory), and, as one agent in a warp
// is enough to make it wait, 53 -> 47 us for the 65,000-agent shared space.  An
// agent with more candidates at nearly one distance than the list holds searches
// again with a sorted list (sorted_search): 40,000 agents at 40 points 64 -> 0.9 ms.
//
// Bound by issue slots in large scenes (0.74 of one instruction a cycle per
// scheduler, 57 % of an instruction's lanes active: the LP's re-solves and the
// half-planes' constructions differ between the lanes; 4 % of the memory's
// rate), by one thread's chain in smaller ones.  1M clusters, one step: 454 us
// with the sorted list in shared memory, 420 with the network and a pass that
// ranks the admitted slots, 394 with the places carried in the entries, 378 with
// the LP's order by all pairs and the penetrations kept for the LP (the
// 65,000-agent shared space: 67, 55, 58, 52), 375 with one construction of the
// cut-off and overlap half-planes, 367 in blocks of two warps, 376 with the sorted
// state read through plain pointers (see wait_for_primary).  (The benchmark's
// 1M crowd after its warm-up steps: 381 -> 304 us.)  Of the 378 the row scan took
// about 90 us, the network 60, the half-planes 58, the LP 130.  Registers, in the
// same form: seven blocks of four warps an SM (72) 380 us and 73 us at 130,000
// agents, six 403 and 88, eight 377 and 76, nine 396 and 79.
#pragma once

#include "orca_step_kernels.cuh"

namespace orca {

__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The N smallest of the sorted D and of a and b.  The i-th smallest of the
// union is min(D[i], max(D[i - 1], x), max(D[i - 2], y)) for x <= y.
template <int N>
__device__ __forceinline__ void insert_pair(float (&D)[N], float a, float b) {
    const float x = fminf(a, b), y = fmaxf(a, b);
#pragma unroll
    for (int i = N - 1; i >= 2; --i) D[i] = min3(D[i], fmaxf(D[i - 1], x), fmaxf(D[i - 2], y));
    D[1] = min3(D[1], fmaxf(D[0], x), y);
    D[0] = fminf(D[0], x);
}

// Shared memory of a warp, in 16-byte units per lane: kl line slots, then kl
// words (the neighbours in order, then each line's penetration at v_A).  The
// search's list of admitted slots lives in the line slots.
__host__ __device__ constexpr int agent_units(int kl) { return kl + (kl + 3) / 4; }

// The two rare paths of the search, kept small (no unrolling, the second out of
// line): with them unrolled in place 1M clusters took 380-455 us instead of 368.

// Puts J[0 .. cnt), the slots of the k nearest, in order by (d^2, index) where
// their entries were equal above the replaced bits (bit m of tied: the m-th and
// the one after it).  A run of ties that goes on beyond the k-th is chosen from
// the list first.
__device__ __forceinline__ void order_ties(float2 p, const float2* pos, const uint2* aux, int* raw, int found,
                                           int* J, int cnt, uint32_t tied, uint32_t replaced) {
    auto dist2 = [&](int j) {
        const float2 q = pos[j];
        return key_d2(p.x, p.y, q.x, q.y);
    };
    if ((tied >> (cnt - 1)) & 1u) {
        const int m = 32 - __clz((int)(~tied & ((1u << (cnt - 1) << 1) - 1u)));
        const uint32_t run = __float_as_uint(dist2(J[m * 32])) & ~replaced;
        int members = 0;
#pragma unroll 4
        for (int e = 0; e < found; ++e) {
            const int j = raw[e * 32];
            if ((__float_as_uint(dist2(j)) & ~replaced) == run) raw[32 * members++] = j;
        }
#pragma unroll 1
        for (int at = m; at < cnt; ++at) {   // the first of those left, each time
            int best = 0, jb = raw[0], ob = aux_orig(aux[jb]);
            float db = dist2(jb);
#pragma unroll 1
            for (int e = 1; e < members; ++e) {
                const int j = raw[e * 32];
                const float d = dist2(j);
                const int o = aux_orig(aux[j]);
                if (d < db || (d == db && o < ob)) {
                    best = e;
                    jb = j;
                    db = d;
                    ob = o;
                }
            }
            J[at * 32] = jb;
            raw[best * 32] = raw[--members * 32];
        }
        tied &= (1u << m) - 1u;
    }
#pragma unroll 1
    for (; tied != 0u; tied &= tied - 1u) {   // insertion sort of every run
        int at = __ffs((int)tied);            // (the second of the pair)
        const int j = J[at * 32];
        const float d = dist2(j);
        const int o = aux_orig(aux[j]);
#pragma unroll 1
        for (; at > 0; --at) {
            const int i = J[(at - 1) * 32];
            const float di = dist2(i);
            if (di < d || (di == d && aux_orig(aux[i]) < o)) break;
            J[at * 32] = i;
        }
        J[at * 32] = j;
    }
}

// Grid rows around an agent: its place in them and their lower bounds of dy^2.
struct Rows {
    const uint32_t* cs;
    int cx, cy, nx, ny;
    float ch, mg, pry, fx;
};

// The search with a sorted list (slots in J, keys in key and orig), for agents
// with more candidates at nearly one distance than the list of slots holds.
__device__ __noinline__ int sorted_search(float2 p, int s, int k, float lim, Rows g,
                                          const float2* pos, const uint2* aux, int* J, float* key,
                                          int* orig) {
    int cnt = 0;
    // candidate j: into the list when before its last entry, the ones behind it shift
    auto consider = [&](int j, float d2, int oj) {
        if (!(d2 <= lim) || (cnt == k && d2 == lim && oj > orig[(k - 1) * 32])) return;
        int at = min(cnt, k - 1);
        while (at > 0) {
            const float de = key[(at - 1) * 32];
            const int oe = orig[(at - 1) * 32];
            if (de < d2 || (de == d2 && oe < oj)) break;
            key[at * 32] = de;
            orig[at * 32] = oe;
            J[at * 32] = J[(at - 1) * 32];
            --at;
        }
        key[at * 32] = d2;
        orig[at * 32] = oj;
        J[at * 32] = j;
        cnt = min(cnt + 1, k);
        if (cnt == k) lim = key[(k - 1) * 32];
    };
    for (int m = 0;; ++m) {
        bool any = false;
        for (int side = m == 0 ? 1 : 0; side < 2; ++side) {
            const int ry = side == 0 ? g.cy - m : g.cy + m;
            if (ry < 0 || ry >= g.ny) continue;
            const float by0 = ry == 0 ? -CUDART_INF_F : (float)ry * g.ch - g.mg;
            const float by1 = ry == g.ny - 1 ? CUDART_INF_F : (float)(ry + 1) * g.ch + g.mg;
            const float ey = fmaxf(fmaxf(by0 - g.pry, g.pry - by1), 0.0f);
            const float g2 = m == 0 ? 0.0f : ey * ey * 0.99999f;
            if (g2 > lim) continue;
            any = true;
            const uint32_t* c = g.cs + (size_t)ry * g.nx;
            const int rb = (int)c[0], re = (int)c[g.nx];
            const int b = (int)c[g.cx], e = (int)c[g.cx + 1];
            int jr = m == 0 ? s + 1 : min(b + (int)(g.fx * (float)(e - b)), e);
            int jl = m == 0 ? s - 1 : jr - 1;
            bool ron = jr < re, lon = jl >= rb;
            while (ron || lon) {
                float2 qr = p, ql = p;
                int orr = 0, ol = 0;
                if (ron) {
                    qr = pos[jr];
                    orr = aux_orig(aux[jr]);
                }
                if (lon) {
                    ql = pos[jl];
                    ol = aux_orig(aux[jl]);
                }
                if (ron) {
                    const float dx = __fsub_rn(qr.x, p.x), dy = __fsub_rn(qr.y, p.y);
                    const float xx = __fmul_rn(dx, dx);
                    if (dx > 0.0f && __fadd_rn(xx, g2) > lim) {
                        ron = false;
                    } else {
                        consider(jr, __fadd_rn(xx, __fmul_rn(dy, dy)), orr);
                        ron = ++jr < re;
                    }
                }
                if (lon) {
                    const float dx = __fsub_rn(ql.x, p.x), dy = __fsub_rn(ql.y, p.y);
                    const float xx = __fmul_rn(dx, dx);
                    if (dx < 0.0f && __fadd_rn(xx, g2) > lim) {
                        lon = false;
                    } else {
                        consider(jl, __fadd_rn(xx, __fmul_rn(dy, dy)), ol);
                        lon = --jl >= rb;
                    }
                }
            }
        }
        if (!any) return cnt;   // both sides at the edge or beyond the bound
    }
}

// One thread per agent (sorted slot s), k <= KC, the incremental LP.
// MODE_PLAIN, or MODE_RECORD with the LP's active set.  kl: line slots per
// lane (KC, and the kinematic half-planes if the scene has them).
template <class SRC, int MODE, int KC>
__global__ void __launch_bounds__(128, KC <= 10 ? 7 : 1)
agent_solve_kernel(int n, int kl, SRC src, const float2* pos, const float2* vel,
                   const uint2* aux, const uint32_t* cstart, AgentIn ain,
                   const float2* __restrict__ vpd, StepOut out, DebugOut dbg,
                   int* __restrict__ err) {
    extern __shared__ float4 smem_lines[];
    wait_for_primary();
    // after a binning kernel that gave up or found inconsistent counts the
    // sorted state is not valid: leave everything as it is (the status call
    // reports the error)
    if (__ldcg(err) & (ERR_BIT_TIMEOUT | ERR_BIT_STATE)) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned lanes = __ballot_sync(0xffffffffu, s < n);
    if (s >= n) return;
    float4* L = smem_lines + (threadIdx.x >> 5) * agent_units(kl) * 32 + (threadIdx.x & 31);
    int* J = reinterpret_cast<int*>(L - (threadIdx.x & 31) + kl * 32) + (threadIdx.x & 31);
    int* raw = reinterpret_cast<int*>(L - (threadIdx.x & 31)) + (threadIdx.x & 31);
    // low bits of an entry of the network: a place in raw
    constexpr uint32_t kPlace = KC <= 16 ? 63u : 127u;
    const int cap = min(4 * kl, (int)kPlace);   // entries of raw
    const SceneDev& sc = src.get(s);
    const float2 p = pos[s];
    const float2 v = vel[s];
    const uint2 as = aux[s];
    const float r = aux_rad(as);
    const int ta = aux_type(as);
    const int o = aux_orig(as);
    const int cx = cell_axis(p.x, sc.origin_x, sc.inv_cell_x, sc.nx);
    const int cy = cell_axis(p.y, sc.origin_y, sc.inv_cell_y, sc.ny);

    // ---- k nearest by (d^2, index), exact search over the x-sorted grid rows ----
    const int k = sc.k;
    int cnt = 0;
    if (k > 0 && isfinite(p.x) && isfinite(p.y)) {   // (a non-finite state is an error)
        const float R2 = sc.R2;
        // the largest float below R_n^2: a candidate within the bound (this, or
        // the k-th distance once k are known, its low bits set) is admitted,
        // and a row cursor stops beyond it
        float thr0 = R2 > 0.0f ? __int_as_float(__float_as_int(R2) - 1) : -1.0f;
        // sorted; the first KC - k entries are below every distance, the ones
        // not yet found above
        float D[KC + 1];
        auto clear = [&]() {
#pragma unroll
            for (int i = 0; i <= KC; ++i)
                D[i] = i < KC - k ? -1.0f : __uint_as_float(__float_as_uint(thr0) | kPlace);
        };
        auto bound = [&]() {
            return fminf(thr0, __uint_as_float(__float_as_uint(D[KC - 1]) | kPlace));
        };
        auto entry = [](float d2, int place) {
            return __uint_as_float((__float_as_uint(d2) & ~kPlace) | (uint32_t)place);
        };
        clear();
        const uint32_t* cs = cstart + sc.cell_off;
        int found = 0;
        // Every grid row is one run of slots sorted by x (the binning kernel
        // orders each cell by x, and cells of a row are consecutive in x).
        // A row is scanned outward from the agent's x with two cursors: the
        // right one stops at the first candidate right of the agent whose
        // fl(dx^2 + g2) exceeds the bound, the left one likewise on the left,
        // where g2 is the row's lower bound of dy^2; every candidate farther
        // along has a larger dx^2, and d^2 = fl(dx^2 + dy^2) >= fl(dx^2 + g2)
        // (rounding is monotone), so none of them can enter the list.
        // Any start slot is valid (candidates on the wrong side of the agent
        // never stop a cursor); a good start only saves candidate tests.
        // Rows are visited nearest first (the agent's own row, then one row
        // on each side in turn, the nearer of the two first) and a side ends
        // at the first row whose y gap is beyond the bound.
        const int nx = sc.nx, ny = sc.ny;
        const float ch = sc.cell_h, mg = sc.ring_delta * ch;
        const float pry = __fsub_rn(p.y, sc.origin_y);
        // lower bound of dy^2 for every agent binned into row ry (widened by
        // the cell-rounding margin, open toward the grid edge), with the
        // 1e-5 relative slack of the key comparison
        auto row_gap2 = [&](int ry) {
            const float by0 = ry == 0 ? -CUDART_INF_F : (float)ry * ch - mg;
            const float by1 = ry == ny - 1 ? CUDART_INF_F : (float)(ry + 1) * ch + mg;
            const float ey = fmaxf(fmaxf(by0 - pry, pry - by1), 0.0f);
            return ey * ey * 0.99999f;
        };
        // start slot of row ry: the agent's x interpolated inside the row's
        // cell of column cx (x-sorted, so agents spread roughly evenly)
        const float fx = fminf(fmaxf(__fmul_rn(__fsub_rn(p.x, sc.origin_x), sc.inv_cell_x) -
                                         (float)cx, 0.0f), 1.0f);
        // Rows in visiting order, through one copy of the row scan: the agent's
        // own row (ring 0) from its neighbouring slots (the agent itself is
        // never a candidate), then ring by ring the nearer of rows cy - m and
        // cy + m first.
        bool up = true, down = true;   // rows cy + m / cy - m left to visit
        int m = 0, so = 2;             // ring, and the next of its two sides
        float gd = 0.0f, gu = 0.0f;    // the ring's y gaps below and above
        int first = 0;
        int ry = cy, jr = s + 1, jl = s - 1;
        float g2 = 0.0f;
        for (;;) {
            const int rb = (int)cs[ry * nx], re = (int)cs[ry * nx + nx];
            bool ron = jr < re, lon = jl >= rb;
            float2 nr = pos[min(jr, n - 1)], nl = pos[max(jl, 0)];
            while (ron || lon) {
                // the next candidates are on their way while these are tested
                const float2 qr = nr, ql = nl;
                nr = pos[min(jr + 1, n - 1)], nl = pos[max(jl - 1, 0)];
                const float lim = bound();
                const float dxr = __fsub_rn(qr.x, p.x), dxl = __fsub_rn(ql.x, p.x);
                const float xxr = __fmul_rn(dxr, dxr), xxl = __fmul_rn(dxl, dxl);
                ron = ron && !(dxr > 0.0f && __fadd_rn(xxr, g2) > lim);
                lon = lon && !(dxl < 0.0f && __fadd_rn(xxl, g2) > lim);
                const float dyr = __fsub_rn(qr.y, p.y), dyl = __fsub_rn(ql.y, p.y);
                float dr = __fadd_rn(xxr, __fmul_rn(dyr, dyr));
                float dl = __fadd_rn(xxl, __fmul_rn(dyl, dyl));
                if (!(ron && dr <= lim)) dr = CUDART_INF_F;   // (not a number either)
                if (!(lon && dl <= lim)) dl = CUDART_INF_F;
                float er = dr, el = dl;
                if (dr < CUDART_INF_F) {
                    er = entry(dr, found);
                    raw[found++ * 32] = jr;
                }
                if (dl < CUDART_INF_F) {
                    el = entry(dl, found);
                    raw[found++ * 32] = jl;
                }
                insert_pair<KC + 1>(D, er, el);
                ron = ron && ++jr < re;
                lon = lon && --jl >= rb;
                if (found > cap - 2) {
                    // the list is full: the candidates within the bound stay;
                    // should that be most of them, the search starts again
                    const float keep = bound();
                    int kept = 0;
#pragma unroll 1
                    for (int e = 0; e < found; ++e) {
                        const int j = raw[e * 32];
                        const float2 q = pos[j];
                        if (key_d2(p.x, p.y, q.x, q.y) <= keep) raw[32 * kept++] = j;
                    }
                    found = kept;
                    clear();
#pragma unroll 1
                    for (int e = 0; e < found; ++e) {
                        const float2 q = pos[raw[e * 32]];
                        insert_pair<KC + 1>(D, entry(key_d2(p.x, p.y, q.x, q.y), e),
                                            CUDART_INF_F);
                    }
                    if (found > cap / 2) {
                        thr0 = -1.0f;   // (nothing is within the bound any more)
                        ron = lon = false;
                    }
                }
            }
            bool more = false;
            while (!more && (up || down)) {
                if (so == 2) {
                    ++m;
                    so = 0;
                    gd = row_gap2(cy - m);
                    gu = row_gap2(cy + m);
                    first = gu < gd ? 1 : 0;
                }
                const int side = so ^ first;
                ++so;
                if (!(side == 0 ? down : up)) continue;
                ry = side == 0 ? cy - m : cy + m;
                g2 = side == 0 ? gd : gu;
                if (ry < 0 || ry >= ny || g2 > bound()) {
                    if (side == 0) down = false;
                    else up = false;
                    continue;
                }
                more = true;
            }
            if (!more) break;
            const int c = ry * nx + cx;
            const int b = (int)cs[c], e = (int)cs[c + 1];
            jr = min(b + (int)(fx * (float)(e - b)), e);
            jl = jr - 1;
        }
        if (thr0 < 0.0f && R2 > 0.0f) {
            cnt = sorted_search(p, s, k, __int_as_float(__float_as_int(R2) - 1),
                                Rows{cs, cx, cy, nx, ny, ch, mg, pry, fx}, pos, aux,
                                J, reinterpret_cast<float*>(raw), raw + kl * 32);
        } else {
            cnt = min(found, k);
            // the neighbours in order: entry KC - k + m is the m-th, unless entries
            // that follow one another differ in the replaced bits only
            const int fill = KC - k;
            uint32_t tied = 0u;
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                const uint32_t a = __float_as_uint(D[i]), b = __float_as_uint(D[i + 1]);
                const int at = i - fill;
                if (at >= 0 && at < cnt) {
                    J[at * 32] = raw[(int)(a & kPlace) * 32];
                    if ((a ^ b) <= kPlace && at + 1 < found) tied |= 1u << at;
                }
            }
            if (tied != 0u) order_ties(p, pos, aux, raw, found, J, cnt, tied, kPlace);
        }
    }
    __syncwarp(lanes);   // the lines take the place of the lists

    // ---- preferred velocity toward the goal or the current waypoint ----
    float2 g = ain.goal[o];
    const float vmax = ain.max_speed[o];
    if (ain.route != nullptr) {
        const int rt = ain.route[o];
        if (rt >= 0) {
            int wi = ain.wp_idx[o];
            if (dbg.swp != nullptr) dbg.swp[o] = (uint8_t)wi;
            wi = advance_waypoint(ain.waypoints + (size_t)rt * ain.n_waypoints, ain.n_waypoints,
                                  wi, p, r, g);
            ain.wp_idx[o] = (uint8_t)wi;
            if (dbg.wp_used != nullptr) dbg.wp_used[o] = (uint8_t)wi;
        }
    }
    const float2 vp = preferred_velocity(p, g, vmax, sc.inv_dt, vpd != nullptr,
                                         vpd != nullptr ? vpd[o] : make_float2(0.0f, 0.0f));

    // ---- one ORCA half-plane per neighbour (Sec. 3.1) ----
    // Constraint m is the m-th nearest.  pen[m], its penetration at v_A, takes
    // the place of the neighbour's slot.
    if (dbg.nbr != nullptr) {
        int32_t* nb = dbg.nbr + (size_t)o * dbg.k_stride;
        for (int m = 0; m < dbg.k_stride; ++m)
            nb[m] = m < cnt ? aux_orig(aux[J[m * 32]]) : -1;
    }
    float* pen = reinterpret_cast<float*>(J);
    bool any_overlap = false;
    uint32_t capbits = 0u, ovbits = 0u;   // per-line construction (MODE_RECORD)
    int nlines = 0;
    // the two lines most violated at v_A so far
    float pm0 = -CUDART_INF_F, pm1 = -CUDART_INF_F;
    int im0 = -1, im1 = -1;
    auto add_line = [&](float4 l) {
        const float pv = penetration(l, v.x, v.y);
        L[nlines * 32] = l;
        pen[nlines * 32] = pv;
        if (pv > pm0) {
            pm1 = pm0;
            im1 = im0;
            pm0 = pv;
            im0 = nlines;
        } else if (pv > pm1) {
            pm1 = pv;
            im1 = nlines;
        }
        ++nlines;
    };
    for (int i = 0; i < cnt; ++i) {
        const int j = J[i * 32];
        const float2 pj = pos[j], vj = vel[j];
        const uint2 aj = aux[j];
        const float rj = aux_rad(aj);
        const int tb = aux_type(aj);
        const float rs = __fadd_rn(r, rj);
        const bool ov = key_d2(p.x, p.y, pj.x, pj.y) <= __fmul_rn(rs, rs);
        any_overlap |= ov;
        const float f = tb ? (ta ? sc.f11 : sc.f01) : (ta ? sc.f10 : sc.f00);
        bool cap_line;
        add_line(orca_line(p.x, p.y, v.x, v.y, r, pj.x, pj.y, vj.x, vj.y, rj, f, sc.inv_tau,
                           sc.inv_dt, ov, cap_line));
        if (MODE == MODE_RECORD) {
            ovbits |= (ov ? 1u : 0u) << i;
            capbits |= (cap_line ? 1u : 0u) << i;
        }
    }

    // ---- vehicles' kinematic half-planes (off unless the scene sets limits) ----
    if (ta != 0 && (sc.kin_turn || sc.kin_accel)) limit_lines(sc, v, vp, add_line);

    // ---- constraint order of the LP ----
    // Half-planes in decreasing penetration at the agent's current velocity:
    // the least-penetration optimum usually rests on the most violated ones,
    // so fewer of the later lines force a re-solve.  The two most violated
    // go first (swaps: slot 0 <-> sw0, then slot 1 <-> sw1); with at most 16
    // lines the rest follow in sorted order (ties keep their order).  The LP's
    // result does not depend on the order beyond rounding; the recorded
    // active set is mapped back to the neighbour order below, through perm
    // (slot -> neighbour index, 4 bits per slot) when sorted.
    int sw0 = 0, sw1 = 1;
    auto swap_lines = [&](int a, int b) {
        const float4 l = L[a * 32];
        const float q = pen[a * 32];
        L[a * 32] = L[b * 32];
        pen[a * 32] = pen[b * 32];
        L[b * 32] = l;
        pen[b * 32] = q;
    };
    if (nlines > 1) {
        if (im0 > 0) {
            swap_lines(0, im0);
            sw0 = im0;
        }
        if (im1 >= 0 && nlines > 2) {
            const int b = im1 == 0 ? sw0 : im1;   // where the second line is now (>= 1)
            if (b > 1) {
                swap_lines(1, b);
                sw1 = b;
            }
        }
    }
    auto nib = [](uint64_t q, int i) { return (uint32_t)((q >> (4 * i)) & 15ull); };
    auto put = [](uint64_t q, int i, uint32_t x) {
        return (q & ~(15ull << (4 * i))) | ((uint64_t)x << (4 * i));
    };
    uint64_t perm = 0ull;
    if (MODE == MODE_RECORD && nlines <= 16) {
        perm = 0xFEDCBA9876543210ull;
        const uint32_t a0 = nib(perm, sw0);
        perm = put(put(perm, sw0, nib(perm, 0)), 0, a0);
        const uint32_t a1 = nib(perm, sw1);
        perm = put(put(perm, sw1, nib(perm, 1)), 1, a1);
    }
    constexpr int R = 8;
    float q[R];
    bool by_pairs = KC <= 10 && nlines <= 10;
    if (by_pairs) {
        float sum = 0.0f;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            q[u] = u + 2 < nlines ? pen[(u + 2) * 32] : -CUDART_INF_F;
            sum += q[u];
        }
        by_pairs = sum == sum;   // (a penetration that is no number has no rank)
    }
    if (by_pairs) {
        // the rank of each line among slots 2 .. 9, by all pairs (no branches)
        int at[R];
#pragma unroll
        for (int u = 0; u < R; ++u) at[u] = 2;
#pragma unroll
        for (int u = 0; u < R; ++u)
#pragma unroll
            for (int w = u + 1; w < R; ++w) {
                if (q[w] > q[u]) ++at[u];
                else ++at[w];
            }
        float4 l[R];
#pragma unroll
        for (int u = 0; u < R; ++u) l[u] = L[(u + 2) * 32];
        const uint64_t was = perm;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            L[at[u] * 32] = l[u];
            pen[at[u] * 32] = q[u];
            if (MODE == MODE_RECORD) perm = put(perm, at[u], nib(was, u + 2));
        }
    } else if (nlines <= 16) {   // insertion sort
        for (int m = 3; m < nlines; ++m) {
            const float4 e = L[m * 32];
            const float pe = pen[m * 32];
            const uint32_t em = MODE == MODE_RECORD ? nib(perm, m) : 0u;
            int at = m;
            while (at > 2 && pen[(at - 1) * 32] < pe) {
                L[at * 32] = L[(at - 1) * 32];
                pen[at * 32] = pen[(at - 1) * 32];
                if (MODE == MODE_RECORD) perm = put(perm, at, nib(perm, at - 1));
                --at;
            }
            L[at * 32] = e;
            pen[at * 32] = pe;
            if (MODE == MODE_RECORD) perm = put(perm, at, em);
        }
    }

    // ---- velocity LP, least-penetration fallback ----
    float vx, vy, tstar;
    uint32_t act = 0u;
    int work = 0;
    const int infeasible =
        solve_velocity(L, 32, nlines, vmax, vp.x, vp.y, v.x, v.y,
                       [&](int i, float4) { return pen[i * 32]; }, vx, vy, tstar, work, act);

    // ---- integrate ----
    const float2 pn = make_float2(__fadd_rn(p.x, __fmul_rn(sc.dt, vx)),
                                  __fadd_rn(p.y, __fmul_rn(sc.dt, vy)));
    const int w = out.caller_order ? o : s;
    out.vel[w] = make_float2(vx, vy);
    out.pos[w] = pn;
    if (out.hint != nullptr) {
        out.hint[s] = (uint32_t)o;
        if (s == 0) *out.hint_ok = 1;
    }
    if (out.key != nullptr) {
        // bin the new position for the next step (as the binning kernel's
        // cell-key phase does on a call's first step)
        const int ncx = cell_axis(pn.x, sc.origin_x, sc.inv_cell_x, sc.nx);
        const int ncy = cell_axis(pn.y, sc.origin_y, sc.inv_cell_y, sc.ny);
        const uint32_t c = (uint32_t)(sc.cell_off + ncy * sc.nx + ncx);
        out.key[s] = c;
        out.slot[s] = atomicAdd(out.count + c, 1u);
    }
    if (dbg.spos != nullptr) dbg.spos[o] = p;
    if (dbg.svel != nullptr) dbg.svel[o] = v;
    if (dbg.vnew != nullptr) dbg.vnew[o] = make_float2(vx, vy);
    if (MODE == MODE_RECORD && dbg.act != nullptr) {
        const int nl = act_nlines(act);
        for (int m = 0; m < nl; ++m) {
            // the LP's line index in the neighbour order
            int li = act_line(act, m);
            if (nlines <= 16) {
                li = (int)nib(perm, li);
            } else {   // undo the two swaps
                li = li == 1 ? sw1 : (li == sw1 ? 1 : li);
                li = li == 0 ? sw0 : (li == sw0 ? 0 : li);
            }
            act = (act & ~(31u << (8 + 8 * m))) | ((uint32_t)li << (8 + 8 * m));
            act |= ((capbits >> li) & 1u) << (13 + 8 * m);
            act |= ((ovbits >> li) & 1u) << (14 + 8 * m);
        }
        dbg.act[o] = act;
    }
    if (dbg.cell != nullptr) dbg.cell[o] = cy * sc.nx + cx;
    if (dbg.cnt != nullptr) dbg.cnt[o] = cnt;
    if (dbg.flags != nullptr) dbg.flags[o] = (uint8_t)(infeasible | (any_overlap ? 4 : 0));
    if (dbg.tstar != nullptr) dbg.tstar[o] = tstar;
}

}  // namespace orca
