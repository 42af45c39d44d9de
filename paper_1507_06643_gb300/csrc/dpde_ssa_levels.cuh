// dpde_ssa_levels.cuh -- the SSA sequence of every domain (Sec. III.A.2,
// III.B.2) executed by dependency levels, domain by domain, each domain's
// state held in shared memory.
//
// The SSA pair map of Eq. (SSA_ij) reads and writes the state of its two
// particles only, so two maps on disjoint particles commute exactly: the
// result of the sequence depends only on, for every particle, the order of
// the maps that touch it. Give map k of the sequence the level
//     lev(k) = 1 + max(lev of the last earlier map touching s_k,
//                      lev of the last earlier map touching t_k)
// (0 if none). Maps of one level touch disjoint particles, and running the
// levels in increasing order keeps, for every particle, the sequence order
// of its maps -- so the level-by-level execution is the sequence, bit for
// bit. At density 3 a domain of ~700 particles has ~3,600 maps in ~100
// levels (the per-class chains of the colour order are ~300 maps deep).
//
// Two kernels per step:
//   k_ssa_sched  one block per domain: stages the domain's forward entries
//                (partner slots, as the force pass wrote them) in shared
//                memory, walks the colour classes in order computing every
//                map's level (a thread per cell of the class: cells of one
//                class share no particle), then sorts the entries by level
//                into records (s, t, w) in global memory.
//   k_ssa_exec   one block per domain: stages (p, eps, id) of the domain,
//                then runs the levels in order, one thread per map. Half of
//                its warps only draw the pairs' Gaussians (Philox is keyed on
//                the ids) in record order, a chunk ahead of the others, which
//                only apply maps, with a barrier of their own between levels.
// Domains too large for the regular shared-memory capacities are deferred to
// a second launch of each kernel with ~2.5x larger capacities (several
// blocks per SM), and from there to a third with what ~200 KB hold; beyond
// those, the execution runs on the state in global memory (same levels, same
// bits), and a domain whose schedule does not fit at all is executed class by
// class along the colour order itself.
#pragma once

#include "dpde_kernels.cuh"

namespace dpde {

// levels of one domain kept by the schedule: 1023, and up to 4095 for whole
// replicas with long rows (Lennard-Jones: 343 particles have ~830 levels,
// 1,000 ~1,120; a schedule that did not fit ran its domain in colour order on
// one block, 11.5 ms a step against 0.8 now; 1,216 replicas of 500 21.6 against
// 2.6)
constexpr int SSA_MAXLEV = 1023, SSA_MAXLEV_LONG = 4095;
constexpr int SCHED_THREADS = 128;
constexpr int SSA_ROW_BATCH = 8;        // entries of a row taken together
constexpr int SSA_LEV_BATCH = 8;        // ... by the level walk
constexpr int SSA_LONG_ROW = 12;        // mean entries of a row from which a warp walks a cell
constexpr int SSA_DRAW_THREADS = 64;    // threads of an execution block that draw Gaussians
constexpr int SSA_EXEC_THREADS_MAX = SSA_THREADS_MAX + SSA_DRAW_THREADS;
constexpr int SSA_CHUNK = 128;          // records drawn ahead of the maps, SSA_RING chunks held
constexpr int SSA_RING = 3;
constexpr int SSA_LOCAL_MAX = 65535;      // particles (and entries) of one domain: 16-bit local indices
constexpr int SSA_NLISTS = 5;             // deferred-domain lists of one step (see enqueue_ssa_levels)

// Domains of the SSA sequence: the cells of each domain sorted by colour
// class (`cells`), the NCOLOURS + 1 class starts of every domain in `cells`
// (`off`), and the first cell of every domain, then the total cell count
// (`cell0`). A domain is a contiguous cell (and slot) range.
struct SsaDomains {
    const int* cells;
    const int* off;
    const int* cell0;
    int n;
};

// The level schedule of every domain: per domain the record offsets of its
// levels (lv_off[d * stride + l], l = 0..nlev, records of level l in
// [lv_off[l], lv_off[l + 1])), its level count (lv_n[d]: nlev >= 0 from the
// regular launch, -3 - nlev from a deferred one, -1 no schedule (executed
// along the colour order), SSA_PENDING = -2 deferred and not yet scheduled),
// and the records, domain d's at [slot0(d) * cap, ...): (s_local | t_local
// << 16) and the weight w, one 8- or 16-byte word. Every domain with lv_n < 0
// is on the list of those the regular schedule deferred and is executed from
// that list, by the deferred launches. The execution's regular launch, which
// may run beside them and beside the schedule's deferred launches, takes only
// lv_n >= 0: no domain is executed twice, and no schedule is read that is
// still being written.
template <class T> struct __align__(2 * sizeof(T)) SsaRec {
    uint32_t st;
    T w;
};

template <class T>
struct SsaLevels {
    int* lv_off;
    int* lv_n;
    SsaRec<T>* rec;
    int stride;   // the most levels + 2
};

// shared bytes of k_ssa_sched for scap particles, ecap entries, ccap cells and
// a level stride: cnt (counters of levels 0..stride - 1, one more) | cr[ccap] (the domain's
// cells in class order: local start | count << 16) | rowoff[scap + 1] |
// L[scap] | ent[ecap] (16-bit)
__host__ __device__ constexpr size_t ssa_sched_smem(int scap, int ecap, int ccap, int stride) {
    return (size_t)(stride + 1 + ccap) * sizeof(int) +
           (((size_t)(2 * scap + 1 + ecap) * 2 + 15) / 16) * 16;
}
// shared bytes of k_ssa_exec for scap staged particles (a multiple of 4): p |
// drawn (G, w) of the chunks held | eps | id | their records | level starts
template <class T>
__host__ __device__ constexpr size_t ssa_exec_smem(int scap, int stride) {
    return (size_t)scap * (sizeof(vec_t<T>) + sizeof(eps_t<T>) + sizeof(uint32_t)) +
           (size_t)SSA_RING * SSA_CHUNK * (sizeof(vec_t<T>) + sizeof(uint32_t)) + (size_t)stride * 2 + 16;
}

// slot range [sb, se) of domain d
template <class T>
__device__ __forceinline__ void ssa_domain_range(const Ctx<T>& C, const SsaDomains& D, int d, int& sb, int& se) {
    sb = C.start[D.cell0[d]];
    se = C.start[D.cell0[d + 1]];
}

// Exclusive scan over n values v(i) held nowhere in particular: each thread
// takes a contiguous run; writes out[i] (16-bit) for i < n and returns the
// total. v is a callable.
template <class F>
__device__ __forceinline__ int block_scan_runs(int n, unsigned short* out, int* sh, F&& v) {
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int i0 = min(n, (int)threadIdx.x * per), i1 = min(n, i0 + per);
    int run = 0;
    for (int i = i0; i < i1; ++i) run += v(i);
    int total;
    int ex = block_exclusive_scan(run, sh, total);
    for (int i = i0; i < i1; ++i) {
        const int x = v(i);
        out[i] = (unsigned short)ex;
        ex += x;
    }
    return total;
}

// The forward entries of the domain's particles, a thread per particle (so a
// warp's lanes read consecutive words of each entry row) with SSA_ROW_BATCH
// loads in flight. use(i, e, v, ok) gets entry e of the domain, of particle
// i, whose row starts at rowoff[i]; past a row's end the last entry again,
// with ok = false, so that nothing branches. fe: entry row 0 of the domain's
// particles.
template <class T, class Use>
__device__ __forceinline__ void ssa_rows(int nb, const unsigned short* rowoff, const ListEnt<T>* fe, size_t N, Use&& use) {
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const int e0 = rowoff[i], n = rowoff[i + 1] - e0;
        const ListEnt<T>* row = fe + i;
        for (int m = 0; m < n; m += SSA_ROW_BATCH) {
            ListEnt<T> v[SSA_ROW_BATCH];
#pragma unroll
            for (int k = 0; k < SSA_ROW_BATCH; ++k) v[k] = row[(size_t)min(m + k, n - 1) * N];
#pragma unroll
            for (int k = 0; k < SSA_ROW_BATCH; ++k) use(i, e0 + min(m + k, n - 1), v[k], m + k < n);
        }
    }
}

// One domain's schedule on the calling block. Returns false (nothing written)
// when the domain exceeds scap particles, ecap entries or the levels kept.
template <class T>
__device__ bool ssa_sched_domain(const Ctx<T>& C, const SsaDomains& D, const SsaLevels<T>& V, int d, int scap,
                                 int ecap, int ccap, bool deferred, unsigned char* smem) {
    __shared__ int sh[32];
    __shared__ int s_flag, s_nlev;
    __shared__ int s_off[NCOLOURS + 1];
    int sb, se;
    ssa_domain_range(C, D, d, sb, se);
    const int nb = se - sb;
    const int tid = threadIdx.x;
    if (nb > scap || nb > SSA_LOCAL_MAX) return false;
    int* cnt = reinterpret_cast<int*>(smem);
    unsigned int* cr = reinterpret_cast<unsigned int*>(cnt + V.stride + 1);
    unsigned short* rowoff = reinterpret_cast<unsigned short*>(cr + ccap);
    unsigned short* L = rowoff + scap + 1;
    unsigned short* ent = L + scap;    // partner (local slot) of each entry, then its level
    if (tid == 0) {
        s_flag = 0;
        s_nlev = 0;
    }
    for (int l = tid; l <= V.stride; l += blockDim.x) cnt[l] = 0;
    const int* off = D.off + (size_t)d * (NCOLOURS + 1);
    for (int k = tid; k <= NCOLOURS; k += blockDim.x) s_off[k] = __ldg(off + k);
    __syncthreads();
    // the domain's cells in class order, start and particle count, read once
    // here rather than class by class in the walk (a domain with more cells
    // than ccap reads them in the walk)
    const int cbase = s_off[0], ncell = s_off[NCOLOURS] - cbase;
    const bool cstaged = ncell <= ccap;
    if (cstaged)
        for (int u = tid; u < ncell; u += blockDim.x) {
            const int c = __ldg(D.cells + cbase + u);
            const int a = C.start[c], b = C.start[c + 1];
            cr[u] = (unsigned int)(a - sb) | ((unsigned int)(b - a) << 16);
        }
    // 1. row offsets of the domain's forward entries (16-bit: checked below)
    for (int i = tid; i < nb; i += blockDim.x) L[i] = (unsigned short)C.fwd_n[sb + i];
    __syncthreads();
    const int E = block_scan_runs(nb, rowoff, sh, [&](int i) { return (int)L[i]; });
    if (E > ecap || E > SSA_LOCAL_MAX) return false;   // uniform over the block
    if (tid == 0) rowoff[nb] = (unsigned short)E;
    __syncthreads();   // the row lengths have been read
    for (int i = tid; i < nb; i += blockDim.x) L[i] = 0;
    __syncthreads();   // the rows' offsets were written by other threads
    const size_t N = (size_t)C.N;
    const ListEnt<T>* fe = C.fwd + sb;   // entry m of local particle i at fe[m N + i]
    // 2. partner slots, local
    ssa_rows(nb, rowoff, fe, N, [&](int, int e, const ListEnt<T>& v, bool) {
        const int t = v.j - sb;
        if ((unsigned)t >= (unsigned)nb) s_flag = 1;   // never by construction
        ent[e] = (unsigned short)min(max(t, 0), nb - 1);
    });
    __syncthreads();
    if (s_flag) {
        if (tid == 0) flag(C.status, ST_DOMAIN);
        return false;
    }
    // 3. levels, class by class, a thread per cell (the cells of a class
    //    share no particle) walking its rows -- the cell's particles in slot
    //    order -- a batch of entries at a time: the partners of a row are
    //    distinct particles, so their levels are loaded at once and only the
    //    recurrence lev_j = 1 + max(lev_{j-1}, L[t_j]) is serial. (Eight lanes
    //    a cell and a prefix maximum over them took 29,000 warp instructions
    //    a domain. Schedule of a step, with the rows below loaded without
    //    branches: 4M 523 -> 417 us, the batch of 256 boxes 1078 -> 826 us.)
    //    Long rows (Lennard-Jones: ~26 entries, 13 particles a cell) come with
    //    few cells a class, one or two of a block's threads walking while the
    //    others wait: there a warp takes a cell, 32 entries of a row at a time
    //    by a prefix maximum (schedule of a step: 343 Lennard-Jones particles
    //    180 -> 112 us, 125 domains of 1,152 278 -> 192).
    const bool long_rows = E > SSA_LONG_ROW * nb;   // uniform over the block
    int mylev = 0;
    for (int k = 0; k < NCOLOURS; ++k) {
        const int k0 = s_off[k], k1 = s_off[k + 1];
        if (k1 == k0) continue;   // uniform over the block
        auto cell_range = [&](int u, int& i, int& iend) {
            if (cstaged) {
                const unsigned int v = cr[u - cbase];
                i = (int)(v & 0xffffu);
                iend = i + (int)(v >> 16);
            } else {
                const int c = __ldg(D.cells + u);
                i = C.start[c] - sb;
                iend = C.start[c + 1] - sb;
            }
        };
        if (long_rows) {
            for (int u = k0 + (tid >> 5); u < k1; u += (int)blockDim.x >> 5) {
                const int lane = tid & 31;
                int i, iend;
                cell_range(u, i, iend);
                for (; i < iend; ++i) {
                    const int end = rowoff[i + 1];
                    int Ls = L[i];
                    for (int e = rowoff[i]; e < end; e += 32) {
                        // lev_j = max(Ls + 1 + j, max over m <= j of L[t_m] + 1 + j - m)
                        const int f = min(e + lane, end - 1), t = ent[f];
                        int x = max((int)L[t], lane == 0 ? Ls : 0) + 1 - lane;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, x, o);
                            if (lane >= o) x = max(x, y);
                        }
                        x += lane;
                        if (e + lane < end) {
                            L[t] = (unsigned short)x;
                            ent[f] = (unsigned short)x;
                        }
                        Ls = __shfl_sync(0xffffffffu, x, min(31, end - 1 - e));
                    }
                    if (lane == 0) L[i] = (unsigned short)Ls;
                    mylev = max(mylev, Ls);
                    __syncwarp();   // the next row reads these levels
                }
            }
            __syncthreads();
            continue;
        }
        for (int u = k0 + tid; u < k1; u += blockDim.x) {
            int i, iend;
            cell_range(u, i, iend);
            int e = i < iend ? rowoff[i] : 0;
            for (; i < iend; ++i) {
                const int end = rowoff[i + 1];
                int Ls = L[i];
                for (; e < end; e += SSA_LEV_BATCH) {
                    // (past the row's end: its last entry again, which
                    // changes nothing)
                    int t[SSA_LEV_BATCH], l[SSA_LEV_BATCH];
#pragma unroll
                    for (int b = 0; b < SSA_LEV_BATCH; ++b) t[b] = ent[min(e + b, end - 1)];
#pragma unroll
                    for (int b = 0; b < SSA_LEV_BATCH; ++b) l[b] = L[t[b]];
#pragma unroll
                    for (int b = 0; b < SSA_LEV_BATCH; ++b) {
                        if (e + b < end) Ls = max(Ls, l[b]) + 1;   // (at most E <= SSA_LOCAL_MAX)
                        l[b] = Ls;
                    }
#pragma unroll
                    for (int b = 0; b < SSA_LEV_BATCH; ++b) {
                        L[t[b]] = (unsigned short)l[b];
                        ent[min(e + b, end - 1)] = (unsigned short)l[b];
                    }
                }
                e = end;
                L[i] = (unsigned short)Ls;
                mylev = max(mylev, Ls);
            }
        }
        __syncthreads();
    }
    atomicMax(&s_nlev, mylev);
    __syncthreads();
    const int nlev = s_nlev;
    if (nlev > V.stride - 2) return false;
    // 4. records sorted by level: counts, offsets, scatter
    for (int e = tid; e < E; e += blockDim.x) atomicAdd(cnt + ent[e], 1);
    __syncthreads();
    int* lvo = V.lv_off + (size_t)d * V.stride;
    if (tid < 32) {
        // exclusive scan of the counts of levels 1..nlev: lvo[l - 1] = start
        // of level l, lvo[nlev] = E; the counters become the cursors
        int carry = 0;
        for (int l0 = 1; l0 <= nlev + 1; l0 += 32) {
            const int l = l0 + tid;
            const int v = l <= nlev ? cnt[l] : 0;
            int x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (tid >= o) x += y;
            }
            if (l <= nlev + 1) {
                lvo[l - 1] = carry + x - v;
                cnt[l] = carry + x - v;
            }
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    // the partners again from the force pass's list (just read: cached), the
    // weights with them
    const size_t base = (size_t)sb * C.nbr_cap;
    ssa_rows(nb, rowoff, fe, N, [&](int i, int e, const ListEnt<T>& v, bool ok) {
        const int pos = atomicAdd(cnt + ent[e], ok ? 1 : 0);
        const SsaRec<T> x{(uint32_t)i | ((uint32_t)min(max(v.j - sb, 0), nb - 1) << 16), v.w};
        if (ok) V.rec[base + pos] = x;
    });
    if (tid == 0) V.lv_n[d] = deferred ? -3 - nlev : nlev;
    return true;
}

// level count of a schedule stored as lv_n (see SsaLevels); -1 without one
__device__ __forceinline__ int ssa_nlev(int v) { return v <= -3 ? -3 - v : v; }

// One launch over the domains. Regular form (list == nullptr): block u takes
// domain d0 + u. Deferred form: the blocks loop over `list`. A domain beyond
// the launch's capacities is passed on to `defer` when one is given (lv_n =
// SSA_PENDING until a later launch schedules it), else left without a
// schedule (lv_n = -1: executed along the colour order).
constexpr int SSA_PENDING = -2;

template <class T>
__global__ void __launch_bounds__(SCHED_THREADS, 8) k_ssa_sched(Ctx<T> C, SsaDomains D, SsaLevels<T> V, int scap,
                                                                 int ecap, int ccap, int d0,
                                                                 const int* __restrict__ list,
                                                                 const int* __restrict__ nlist, int* defer,
                                                                 int* ndefer) {
    extern __shared__ __align__(16) unsigned char sched_smem[];
    const int n = list ? *nlist : (int)gridDim.x;
    for (int u = blockIdx.x; u < n; u += gridDim.x) {
        const int d = list ? list[u] : d0 + u;
        if (!ssa_sched_domain(C, D, V, d, scap, ecap, ccap, list != nullptr, sched_smem) && threadIdx.x == 0) {
            V.lv_n[d] = defer ? SSA_PENDING : -1;
            if (defer) defer[atomicAdd(ndefer, 1)] = d;
        }
        __syncthreads();
    }
}

// The levels of domain d on the state (P, Es, ID), indexed by local slot, by
// nmap threads that apply maps and the block's others, which draw.
//
// What bounds it: a level holds ~36 maps at density 3 and ~105 levels depend
// on one another, so the applying warps are latency bound, ~400 cycles a
// level, while Philox and Box-Muller are two thirds of the instructions and
// depend on nothing. Drawn by the applying threads they ran on partly filled
// warps and inside the levels' critical path; drawn in record order by warps
// of their own, every lane draws, and the other blocks' drawing fills the
// applying warps' waits. Two drawing warps keep up with two applying ones
// (one: 709 us at 4M; three: 568). Execution of a step: 4M 610 -> 516 us, the
// shock tube 1083 -> 782, 125 domains of 864 particles 110 -> 79 us, 1,000
// particles in FP64 708 -> 321 us.
// the block's barrier, for warps at different places of the code
__device__ __forceinline__ void block_bar() { asm volatile("bar.sync 0;" ::: "memory"); }

template <class T>
__device__ __forceinline__ void ssa_exec_levels(const Ctx<T>& C, const SsaLevels<T>& V, int d, int sb, int rep,
                                                vec_t<T>* P, eps_t<T>* Es, const uint32_t* ID, vec_t<T>* ring,
                                                uint32_t* ring_st, const unsigned short* lvs, int nlev, int nmap,
                                                T dt, T sqrt_dt) {
    static_assert(SSA_THREADS_MAX <= SSA_CHUNK, "see the ring");
    RepInfo R;   // (in registers: the barriers would have a reference read again)
    R.cv = C.reps[rep].cv;
    R.cvf = C.reps[rep].cvf;
    const int tid = threadIdx.x;
    const int E = lvs[nlev];
    const int nchunk = (E + SSA_CHUNK - 1) / SSA_CHUNK;
    const SsaRec<T>* rec = V.rec + (size_t)sb * C.nbr_cap;
    const T amp0 = T(2) * C.sigma * sqrt_dt;   // amplitude of the map as gamma -> 0
    const T k2 = T(2) * dt * C.inv_m;
    if (tid >= nmap) {
        // a record of every SSA_DRAW_THREADS, the next one loaded while this
        // one's Gaussian is drawn
        const uint32_t step = (uint32_t)*C.step;
        int r = tid - nmap;
        SsaRec<T> x{0u, T(0)};
        if (r < E) x = rec[r];
        for (int c = 0; c <= nchunk; ++c) {
            const int end = min(E, (c + 1) * SSA_CHUNK);
            int at = c % SSA_RING * SSA_CHUNK + tid - nmap;
#pragma unroll 1
            for (; r < end; r += SSA_DRAW_THREADS, at += SSA_DRAW_THREADS) {
                const SsaRec<T> y = x;
                if (r + SSA_DRAW_THREADS < E) x = rec[r + SSA_DRAW_THREADS];
                const T3<T> G = pair_gauss<T>(C.seed, step, (uint32_t)rep, ID[y.st & 0xffffu], ID[y.st >> 16]);
                vec_t<T> g;
                g.x = G.x; g.y = G.y; g.z = G.z; g.w = y.w;
                ring[at] = ssa_noise(C, g, k2, amp0);
                ring_st[at] = y.st;
            }
            block_bar();
        }
        return;
    }
    // level ends: the current level's, and the next one's, read a step ahead
    int l = 1, lend = lvs[min(1, nlev)], lnext = lvs[min(2, nlev)];
    block_bar();                           // chunk 0 is drawn
    // Chunk c is drawn while the maps of the records before it run: whole
    // levels, and full steps of a level that reaches into chunk c, so at most
    // nmap - 1 < SSA_CHUNK records of the chunks before are left for later and
    // three chunks hold all that is in use.
    int r = 0, at = 0;   // first record of the step, and its place in the ring
    for (int c = 1; c <= nchunk; ++c) {
        const int avail = min(E, c * SSA_CHUNK);
        auto width = [&](int from) {   // maps of the step at record `from`; 0: not drawn yet, or none left
            const int n = min(lend - from, nmap);
            return from + n <= avail ? n : 0;
        };
        auto load = [&](int n, int a, uint32_t& st, vec_t<T>& g) {
            if (tid < n) {
                int k = a + tid;
                k -= k >= SSA_RING * SSA_CHUNK ? SSA_RING * SSA_CHUNK : 0;
                st = ring_st[k];
                g = ring[k];
            }
        };
        int n = width(r);
        uint32_t st = 0;
        vec_t<T> g{};
        load(n, at, st, g);
        while (n > 0) {
            // the next step and its record, loaded ahead
            r += n;
            at += n;
            at -= at >= SSA_RING * SSA_CHUNK ? SSA_RING * SSA_CHUNK : 0;
            if (r == lend) {
                lend = lnext;
                ++l;
                lnext = lvs[min(l + 1, nlev)];
            }
            const int n2 = width(r);
            uint32_t st2 = 0;
            vec_t<T> g2{};
            load(n2, at, st2, g2);
            if (tid < n) {
                const int s = (int)(st & 0xffffu), t = (int)(st >> 16);
                vec_t<T> ps = P[s];
                eps_t<T> es = Es[s];
                T bs = ps.w;
                vec_t<T> pt = P[t];
                eps_t<T> et = Es[t];
                ssa_noise_map(C, R, ps, es, bs, pt, et, g, k2, amp0);
                ps.w = bs;
                P[s] = ps;
                Es[s] = es;
                P[t] = pt;
                Es[t] = et;
            }
            // the applying threads meet (barrier 1; 0 is the block's)
            asm volatile("bar.sync 1, %0;" ::"r"(nmap) : "memory");
            n = n2;
            st = st2;
            g = g2;
        }
        block_bar();
    }
}

// Domain d without a schedule: its colour classes in order on the state in
// global memory, a thread per cell of the class (the colour order itself).
template <class T>
__device__ void ssa_exec_classes(const Ctx<T>& C, const SsaDomains& D, int d, int rep, T dt, T sqrt_dt) {
    const RepInfo& R = C.reps[rep];
    const T amp0 = T(2) * C.sigma * sqrt_dt;
    const T k2 = T(2) * dt * C.inv_m;
    const uint32_t step = (uint32_t)*C.step;
    const size_t N = (size_t)C.N;
    const int* off = D.off + (size_t)d * (NCOLOURS + 1);
    for (int k = 0; k < NCOLOURS; ++k) {
        const int k0 = off[k], k1 = off[k + 1];
        if (k1 == k0) continue;
        for (int u = k0 + threadIdx.x; u < k1; u += blockDim.x) {
            const int c = D.cells[u];
            for (int s = C.start[c]; s < C.start[c + 1]; ++s) {
                const int nf = C.fwd_n[s];
                if (nf == 0) continue;
                vec_t<T> ps = C.pB[s];
                eps_t<T> es = C.eB[s];
                T bs = ps.w;
                const uint32_t ids = C.idB[s];
                for (int m = 0; m < nf; ++m) {
                    const ListEnt<T> en = C.fwd[(size_t)m * N + s];
                    const int t = en.j;
                    const T3<T> G = pair_gauss<T>(C.seed, step, (uint32_t)rep, ids, C.idB[t]);
                    vec_t<T> g;
                    g.x = G.x;
                    g.y = G.y;
                    g.z = G.z;
                    g.w = en.w;
                    vec_t<T> pt = C.pB[t];
                    eps_t<T> et = C.eB[t];
                    ssa_pair_map(C, R, ps, es, bs, pt, et, g, k2, amp0);
                    C.pB[t] = pt;
                    C.eB[t] = et;
                }
                ps.w = bs;
                C.pB[s] = ps;
                C.eB[s] = es;
            }
        }
        __syncthreads();
    }
}

// One domain on the calling block: staged in shared memory when it fits in
// scap slots, else deferred (defer given) or run on global memory (defer ==
// nullptr). The regular launch skips the domains the regular schedule
// deferred, whether or not a later launch could schedule them.
template <class T>
__device__ void ssa_exec_domain(const Ctx<T>& C, const SsaDomains& D, const SsaLevels<T>& V, int d, int scap,
                                bool regular, int* defer, int* ndefer, int nmap, T dt, T sqrt_dt, unsigned char* smem) {
    int sb, se;
    ssa_domain_range(C, D, d, sb, se);
    const int nb = se - sb;
    if (nb == 0) return;
    const int v = V.lv_n[d];
    const int rep = C.rep_of_cell[D.cell0[d]];
    // deferred by the regular schedule: scheduled (or left without a schedule)
    // and executed by the deferred launches, perhaps running beside this one
    if (regular && v < 0) return;
    const int nlev = ssa_nlev(v);
    if (nlev < 0) {   // no schedule, even with the largest capacities: the colour order itself
        ssa_exec_classes(C, D, d, rep, dt, sqrt_dt);
        return;
    }
    vec_t<T>* P = reinterpret_cast<vec_t<T>*>(smem);
    vec_t<T>* ring = P + scap;
    eps_t<T>* Es = reinterpret_cast<eps_t<T>*>(ring + SSA_RING * SSA_CHUNK);
    uint32_t* ID = reinterpret_cast<uint32_t*>(Es + scap);
    uint32_t* ring_st = ID + scap;
    unsigned short* lvs = reinterpret_cast<unsigned short*>(ring_st + SSA_RING * SSA_CHUNK);
    if (nb > scap && defer) {
        if (threadIdx.x == 0) defer[atomicAdd(ndefer, 1)] = d;
        return;
    }
    const int* lvo = V.lv_off + (size_t)d * V.stride;
    for (int l = threadIdx.x; l <= nlev; l += blockDim.x) lvs[l] = (unsigned short)lvo[l];
    if (nb > scap) {
        __syncthreads();
        ssa_exec_levels(C, V, d, sb, rep, C.pB + sb, C.eB + sb, C.idB + sb, ring, ring_st, lvs, nlev, nmap, dt, sqrt_dt);
        return;
    }
    // four particles per thread in flight
    for (int i0 = threadIdx.x; i0 < nb; i0 += 4 * blockDim.x) {
        vec_t<T> pv[4];
        eps_t<T> ev[4];
        uint32_t iv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * (int)blockDim.x;
            if (i < nb) {
                pv[u] = C.pB[sb + i];
                ev[u] = C.eB[sb + i];
                iv[u] = C.idB[sb + i];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * (int)blockDim.x;
            if (i < nb) {
                P[i] = pv[u];
                Es[i] = ev[u];
                ID[i] = iv[u];
            }
        }
    }
    __syncthreads();
    ssa_exec_levels(C, V, d, sb, rep, P, Es, ID, ring, ring_st, lvs, nlev, nmap, dt, sqrt_dt);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        C.pB[sb + i] = P[i];
        C.eB[sb + i] = Es[i];
    }
}

// Regular form (list == nullptr): block u takes domain d0 + u, leaving out
// the domains the regular schedule deferred (the deferred launches execute
// them). Deferred form: the blocks loop over `list`. A domain with more than
// scap particles is passed on to `defer` when one is given, else run on the
// state in global memory.
template <class T>
__global__ void __launch_bounds__(SSA_EXEC_THREADS_MAX, sizeof(T) == 4 ? 4 : 2) k_ssa_exec(Ctx<T> C, SsaDomains D, SsaLevels<T> V,
                                                                    int scap, int d0, const int* __restrict__ list,
                                                                    const int* __restrict__ nlist, int* defer,
                                                                    int* ndefer, T dt, T sqrt_dt) {
    extern __shared__ __align__(32) unsigned char exec_smem[];   // (aligned here: computed alignment makes generic accesses)
    const int n = list ? *nlist : (int)gridDim.x;
    for (int u = blockIdx.x; u < n; u += gridDim.x) {
        ssa_exec_domain(C, D, V, list ? list[u] : d0 + u, scap, list == nullptr, defer, ndefer,
                        (int)blockDim.x - SSA_DRAW_THREADS, dt, sqrt_dt, exec_smem);
        __syncthreads();
    }
}

}  // namespace dpde
