// dpde_ssa_cells.cuh -- one colour class of the SSA sequence, a warp per cell
// (ssa_mode 0, and DPDE_SSA on replicas too large for the level form).
//
// The cells of a class share no particle, so the warp that has a cell has all
// particles its pairs reach -- those of the cell and of the 13 cells forward
// of it in its domain, ~42 at density 3 -- to itself: it stages their state in
// shared memory once, runs the cell's maps there and writes back what changed.
//
// What bounds it: latency. A thread per cell (k_ssa_colour) walks its chain
// map by map, ~0.4 us each through loads from L2 that depend on one another,
// and the longest of a class, ~50 maps, is the launch's time. Here the lanes
// hold 32 entries of the sequence at a time, each with its rank among the
// maps of either particle; a map whose ranks are up for both runs, so the rows
// of a cell overlap and 32 entries take ~10 rounds. SSA step of 64,000
// particles 642 -> 406 us, of 20,011 442 -> 280, of 200,000 898 -> 655. Every particle sees its
// maps in sequence order: same bits.
#pragma once

#include "dpde_ssa_levels.cuh"

namespace dpde {

// shared bytes of a warp with room for lcap staged particles (at least 16):
// p | eps | slot | maps done | partners of the round
template <class T>
__host__ __device__ constexpr size_t ssa_cells_smem(int lcap) {
    return (size_t)lcap * (sizeof(vec_t<T>) + sizeof(eps_t<T>) + 3 * sizeof(int));
}

// inclusive sum over the lanes
__device__ __forceinline__ int warp_inclusive(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}
// the first lane whose inclusive sum exceeds f (31 if none)
__device__ __forceinline__ int flat_owner(int incl, int f) {
    int lo = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
        const int v = __shfl_sync(0xffffffffu, incl, lo + st - 1);
        if (v <= f) lo += st;
    }
    return lo;
}

template <class T>
__global__ void __launch_bounds__(32) k_ssa_cells(Ctx<T> C, const int* __restrict__ cells, int whole, int lcap, T dt,
                                                  T sqrt_dt) {
    extern __shared__ __align__(32) unsigned char cells_smem[];
    constexpr uint32_t ALL = 0xffffffffu;
    const int lane = threadIdx.x;
    const int c = cells[blockIdx.x];
    const int b = C.start[c], nb = C.start[c + 1] - b;
    if (nb == 0) return;
    const RepInfo& R = C.reps[C.rep_of_cell[c]];
    // lane q < 14: the slots [a, a + n) of the cell q segments forward, none
    // beyond a wall or the domain
    int a = 0, n = 0;
    if (lane < 14) {
        const int cc = C.cB[b], cx = cell_x(cc), cy = cell_y(cc), cz = cell_z(cc);
        const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2], sg = 13 + lane;
        int x = cx + sg % 3 - 1, y = cy + (sg / 3) % 3 - 1, z = cz + sg / 9 - 1;
        bool use = !(R.walls && z >= nz);
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        z = z >= nz ? z - nz : z;
        if (!whole) {
            const int* bt = brick_tab(C.tab, R);
            use = use && __ldg(bt + x) == __ldg(bt + cx) && __ldg(bt + nx + y) == __ldg(bt + nx + cy) &&
                  __ldg(bt + nx + ny + z) == __ldg(bt + nx + ny + cz);
        }
        if (use) {
            const int o = cell_index(C.tab, R, x, y, z);
            a = C.start[o];
            n = C.start[o + 1] - a;
        }
    }
    const int incl = warp_inclusive(n, lane), tot = __shfl_sync(ALL, incl, 31);
    if (tot > lcap) {   // too many for the shared memory: the chain in global memory
        int* rows = reinterpret_cast<int*>(cells_smem);
        if (lane == 0) ssa_cell_chain(C, c, dt, sqrt_dt, rows, rows + SSA_ROWS, 1, 0);
        return;
    }
    vec_t<T>* P = reinterpret_cast<vec_t<T>*>(cells_smem);
    eps_t<T>* Es = reinterpret_cast<eps_t<T>*>(P + lcap);
    int* slot = reinterpret_cast<int*>(Es + lcap);
    volatile int* done = slot + lcap;   // maps done on each staged particle
    int* part = slot + 2 * lcap;        // entries of the round with it as the partner
    for (int l0 = 0; l0 < tot; l0 += 32) {
        const int l = l0 + lane, o = flat_owner(incl, l);
        const int s = __shfl_sync(ALL, a - (incl - n), o) + l;
        if (l < tot) {
            slot[l] = s;
            P[l] = C.pB[s];
            Es[l] = C.eB[s];
            done[l] = 0;
            part[l] = 0;
        }
    }
    __syncwarp();
    const T amp0 = T(2) * C.sigma * sqrt_dt;
    const T k2 = T(2) * dt * C.inv_m;
    const size_t N = (size_t)C.N, cap = (size_t)C.nbr_cap;
    const uint32_t below = (1u << lane) - 1u;
    // the cell's rows, 32 particles at a time; staged particle r is the cell's r-th
    for (int r0 = 0; r0 < nb; r0 += 32) {
        const int nf = r0 + lane < nb ? C.fwd_n[b + r0 + lane] : 0;
        const int fi = warp_inclusive(nf, lane), total = __shfl_sync(ALL, fi, 31);
        // entry f of the rows: staged index of its owner (-1: none), partner slot, noise
        auto fetch = [&](int f, int& ls, int& t, vec_t<T>& g) {
            const int o = flat_owner(fi, f), k = f - __shfl_sync(ALL, fi - nf, o);
            ls = t = -1;
            if (f < total) {
                ls = r0 + o;
                t = C.fwd[(size_t)k * N + b + ls].j;
                g = ssa_noise(C, C.fwd_g[(size_t)(b + ls) * cap + k], k2, amp0);
            }
        };
        int ls, t;
        vec_t<T> g{};
        fetch(lane, ls, t, g);
        for (int f0 = 0; f0 < total; f0 += 32) {
            // staged index of the partner; a lane without an entry gets one of its own
            int lt = -1 - lane;
#pragma unroll
            for (int q = 0; q < 14; ++q) {
                const int qa = __shfl_sync(ALL, a, q), qn = __shfl_sync(ALL, n, q), qo = __shfl_sync(ALL, incl, q);
                if (t >= 0 && (unsigned)(t - qa) < (unsigned)qn) lt = qo - qn + t - qa;
            }
            bool todo = ls >= 0;
            if (todo && lt < 0) {   // never by construction
                flag(C.status, ST_DOMAIN);
                todo = false;
            }
            // ranks: the entries before mine with my owner or with it as the
            // partner (those of earlier rows: all there are), and those before
            // mine with my partner (as an owner it comes later)
            int rs = 0, rt = 0;
            const uint32_t same_s = __match_any_sync(ALL, todo ? ls : -1 - lane);
            const uint32_t same_t = __match_any_sync(ALL, lt);
            if (todo) atomicAdd(&part[lt], 1);
            __syncwarp();
            if (todo) {
                rs = done[ls] + __popc(same_s & below) + part[ls];
                rt = done[lt] + __popc(same_t & below);
            }
            __syncwarp();
            if (todo) part[lt] = 0;
            // the next entries, while these run
            const int cs = ls, ct = lt;
            const vec_t<T> cg = g;
            fetch(f0 + 32 + lane, ls, t, g);
            // the first entry left is always up: at most 32 rounds
            for (int round = 0; round < 32 && __any_sync(ALL, todo); ++round) {
                const bool up = todo && done[cs] == rs && done[ct] == rt;
                __syncwarp();
                if (up) {
                    vec_t<T> ps = P[cs], pt = P[ct];
                    eps_t<T> es = Es[cs], et = Es[ct];
                    T bs = ps.w;
                    ssa_noise_map(C, R, ps, es, bs, pt, et, cg, k2, amp0);
                    ps.w = bs;
                    P[cs] = ps;
                    Es[cs] = es;
                    P[ct] = pt;
                    Es[ct] = et;
                    done[cs] = rs + 1;
                    done[ct] = rt + 1;
                    todo = false;
                }
                __syncwarp();
            }
        }
    }
    for (int l = lane; l < tot; l += 32)
        if (done[l] > 0) {
            C.pB[slot[l]] = P[l];
            C.eB[slot[l]] = Es[l];
        }
}

}  // namespace dpde
