// dpde_kernels.cuh -- the kernels of one DPDE timestep (templated on the
// precision T of positions, momenta, forces and pair arithmetic).
//
// Buffer roles are fixed per step so that one captured step graph can be
// replayed: the state lives in set A between steps; the cell sort gathers
// A -> B; forces and the FD schemes read B; the FD part writes the new state
// back into A (same cell-sorted slot order).
#pragma once

#include "dpde_device.cuh"

namespace dpde {

// LIST_OBS: no lists and no forces, but each particle's sums of the pair potential and its Laplacian
enum ListMode : int { LIST_NONE = 0, LIST_ALL = 1, LIST_CROSS = 2, LIST_FWD = 3, LIST_OBS = 4 };

// One entry of a neighbour or forward list: the partner's slot and w = 1 -
// r / r_cut, written and read as one 8- or 16-byte word.
template <class T> struct __align__(2 * sizeof(T)) ListEnt {
    int j;
    T w;
};

template <class T> struct Ctx {
    using vec = vec_t<T>;
    using E = eps_t<T>;
    vec* qA; vec* pA; E* eA; int* cA;
    vec* qB; vec* pB; E* eB; int* cB;
    uint32_t* idB;   // compact id copy of set B (for neighbour gathers)
    vec* F; vec* dp;
    T* upot;         // per particle: its share of U at the step's positions, 1/2 sum_j v(r_ij)
    int* key;        // global cell of each slot (A order), written by the drift
    int* tmp;        // slots binned by cell, arbitrary order inside a cell
    int* count;      // per-cell counts (ncells), followed by fill (ncells)
    int* fill;
    int* start;      // ncells + 1 exclusive prefix of count
    ListEnt<T>* nbr; // neighbour list, [k * N + i], nbr_cap rows (fwd follows in the same buffer)
    int* nbr_n;      // entries per particle
    int nbr_cap;
    ListEnt<T>* fwd; // forward pairs of the SSA as the force pass writes them, entry-major
                     //   [k * N + i], in SSA sequence order (segment, id)
    vec* fwd_g;      // (G_it, w) of each entry, particle-major [i * nbr_cap + k] (the SSA
                     //   chains' reading order), drawn before the SSA launches; the level
                     //   records of the SSA by levels; then the SER sweeps' delta p_ij
    int* fwd_n;
    const int* rep_of_slot;
    const int* rep_of_cell;
    const int* brick_rep;
    const int* tab;
    const RepInfo* reps;
    const long long* step;   // device step counter
    WallPos* wall;           // upper wall of each replica for this step's drift
    unsigned int* status;
    int N, ncells;
    T m, inv_m, rc, rc2, inv_rc, a, sigma, sig2_4;
    PotT<T> pot;
    PhiloxKeys seed;   // round keys
};

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
template <class T> __device__ __forceinline__ T tfloor(T x);
template <> __device__ __forceinline__ float tfloor(float x) { return floorf(x); }
template <> __device__ __forceinline__ double tfloor(double x) { return floor(x); }

__device__ __forceinline__ float beta_of(ff e, const RepInfo& R) { return R.cvf / e.hi; }
__device__ __forceinline__ double beta_of(double e, const RepInfo& R) { return R.cv / e; }

__device__ __forceinline__ void flag(unsigned int* st, unsigned int bits) { atomicOr(st, bits); }

template <class V> __device__ __forceinline__ bool finite3(const V& v) {
    return isfinite(v.x) && isfinite(v.y) && isfinite(v.z);
}
__device__ __forceinline__ bool eps_ok(double e) { return e > 0.0; }
__device__ __forceinline__ bool eps_ok(ff e) { return e.hi > 0.0f; }
__device__ __forceinline__ bool eps_finite(double e) { return isfinite(e); }
__device__ __forceinline__ bool eps_finite(ff e) { return isfinite(e.hi) && isfinite(e.lo); }

template <class T>
__device__ __forceinline__ void check_state(unsigned int* st, const vec_t<T>& p, const eps_t<T>& e) {
    if (!eps_ok(e)) flag(st, ST_NEG_EPS);
    if (!finite3(p) || !eps_finite(e)) flag(st, ST_NONFINITE);
}

constexpr int NBR_J_BITS = 27;   // particle count limit 2^27 of a handle

template <class T> __device__ __forceinline__ T trsqrt(T x);
template <> __device__ __forceinline__ float trsqrt(float x) { return rsqrtf(x); }
template <> __device__ __forceinline__ double trsqrt(double x) { return rsqrt(x); }

// offset * l for a cell offset d in {-1, 0, 1}
template <class T> __device__ __forceinline__ T shift(int d, T l) {
    return d == 0 ? T(0) : (d > 0 ? l : -l);
}

// ---------------------------------------------------------------------------
// state in / out
// ---------------------------------------------------------------------------
template <class T>
__global__ void k_load_state(Ctx<T> C, const double* __restrict__ q, const double* __restrict__ p,
                             const double* __restrict__ e, int s0, int s1) {
    const int s = s0 + blockIdx.x * blockDim.x + threadIdx.x;   // slots s0 .. s1 - 1
    if (s >= s1) return;
    const RepInfo& R = C.reps[C.rep_of_slot[s]];
    vec_t<T> qv, pv;
    int c[3];
    T o[3];
    for (int d = 0; d < 3; ++d) {
        double x = q[3 * s + d];
        const bool wall = d == 2 && R.walls;   // a walled z is not periodic: z = L_z stays on the top face
        if (!wall && !(x >= 0.0 && x < R.L[d])) {   // wrap only what lies outside [0, L) (FP64 division is slow)
            x -= R.L[d] * floor(x / R.L[d]);
            if (x >= R.L[d]) x -= R.L[d];
        }
        int cd = (int)(x * R.s[d]);
        cd = cd > R.nc[d] - 1 ? R.nc[d] - 1 : (cd < 0 ? 0 : cd);
        c[d] = cd;
        o[d] = (T)(x - (double)cd * R.ell[d]);
    }
    qv.x = o[0]; qv.y = o[1]; qv.z = o[2];
    set_id(qv, (uint32_t)(s - R.part_off));
    eps_t<T> ev;
    eps_from(e[s], ev);
    pv.x = (T)p[3 * s]; pv.y = (T)p[3 * s + 1]; pv.z = (T)p[3 * s + 2];
    pv.w = beta_of(ev, R);
    C.qA[s] = qv;
    C.pA[s] = pv;
    C.eA[s] = ev;
    C.cA[s] = pack_cell(c[0], c[1], c[2]);
}

// slot of every particle of set A, by global id (part_off + id)
template <class T>
__global__ void k_slot_of_id(Ctx<T> C, int* __restrict__ slot_of) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= C.N) return;
    slot_of[C.reps[C.rep_of_slot[s]].part_off + (int)id_of(C.qA[s])] = s;
}

// the state of set A in id order: one thread per id gathers its slot, so the
// FP64 outputs are written contiguously
template <class T>
__global__ void k_get_state(Ctx<T> C, const int* __restrict__ slot_of, double* __restrict__ q,
                            double* __restrict__ p, double* __restrict__ e, int g0, int g1) {
    const int g = g0 + blockIdx.x * blockDim.x + threadIdx.x;   // ids g0 .. g1 - 1
    if (g >= g1) return;
    const int s = slot_of[g];
    const RepInfo& R = C.reps[C.rep_of_slot[s]];
    if (q) {
        const vec_t<T> qv = C.qA[s];
        const int cc = C.cA[s];
        const int cd[3] = {cell_x(cc), cell_y(cc), cell_z(cc)};
        const double od[3] = {(double)qv.x, (double)qv.y, (double)qv.z};
        for (int d = 0; d < 3; ++d) {
            double x = (double)cd[d] * R.ell[d] + od[d];
            if (!(d == 2 && R.walls)) {   // a walled z is not periodic
                if (x >= R.L[d]) x -= R.L[d];
                else if (x < 0.0) x += R.L[d];
            }
            q[3 * (size_t)g + d] = x;
        }
    }
    if (p) {
        const vec_t<T> pv = C.pA[s];
        p[3 * (size_t)g] = (double)pv.x; p[3 * (size_t)g + 1] = (double)pv.y; p[3 * (size_t)g + 2] = (double)pv.z;
    }
    if (e) e[g] = eps_value(C.eA[s]);
}

// ---------------------------------------------------------------------------
// Verlet first half: p += dt/2 F; q += dt p / m, with the offset moved into
// the neighbouring cell when it leaves [0, l) (periodic cell coordinates).
// Then the cell key and the per-cell count of the sort.
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ void move_axis(T& o, int& c, T l, int nc) {
    if (o >= l || o < T(0)) {
        const T f = tfloor(o / l);
        o -= f * l;
        c += (int)f;
        c %= nc;
        if (c < 0) c += nc;
    }
}

// Along a walled z axis: the drifted offset o of cell c, and its momentum
// p_z, mirrored at the wall z = 0 (z -> -z, p_z -> -p_z) or at the upper wall
// z_w = W.c l + W.o (z -> 2 z_w - z, p_z -> two_mu - p_z, two_mu = 2 m u),
// in cell-relative arithmetic.
template <class T>
__device__ __forceinline__ void wall_axis(T& o, int& c, T& pz, T l, int nc, const WallPos& W, T two_mu) {
    int cu = c;
    T on = o;
    if (on >= l || on < T(0)) {
        const T f = tfloor(on / l);
        on -= f * l;
        cu += (int)f;
        if (on >= l) { on -= l; ++cu; }
    }
    if (cu < 0) {
        cu = -cu - 1;
        on = l - on;
        if (on >= l) { on -= l; ++cu; }
        pz = -pz;
    } else {
        const T ow = (T)W.o;
        if (cu > W.c || (cu == W.c && on > ow)) {
            const T d = (T)(cu - W.c) * l + (on - ow);   // z - z_w > 0
            T o2 = ow - d;
            int c2 = W.c;
            const T f = tfloor(o2 / l);
            o2 -= f * l;
            c2 += (int)f;
            if (o2 >= l) { o2 -= l; ++c2; }
            cu = c2;
            on = o2;
            pz = two_mu - pz;
        }
    }
    // a position exactly on the upper face stays in the top cell
    if (cu >= nc) { cu = nc - 1; on = l; }
    if (cu < 0) { cu = 0; on = T(0); }
    o = on;
    c = cu;
}

// Upper-wall position of every replica for the drift of the current step n:
// z_w = L_z + u (n + 1) dt (L_z for replicas without walls). A wall inside
// the lowest cell layer raises ST_WALL.
template <class T>
__global__ void k_wall_pos(Ctx<T> C, int nrep, double dt) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrep) return;
    const RepInfo& I = C.reps[r];
    WallPos w;
    w.c = I.nc[2];
    w.o = 0.0;
    w.pad = 0;
    if (I.walls && I.wall_u != 0.0) {
        const double zw = I.L[2] + I.wall_u * (double)(*C.step + 1) * dt;
        int c = (int)floor(zw * I.s[2]);
        c = c > I.nc[2] ? I.nc[2] : c;
        double o = zw - (double)c * I.ell[2];
        if (o < 0.0) { --c; o += I.ell[2]; }
        if (c < 1) {
            flag(C.status, ST_WALL);
            c = 1;
            o = 0.0;
        }
        w.c = c;
        w.o = o;
    }
    C.wall[r] = w;
}

template <class T>
__global__ void k_kick_drift_key(Ctx<T> C, T half_dt, T dt, int kick) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= C.N) return;
    const int rep = C.rep_of_slot[s];
    const RepInfo& R = C.reps[rep];
    int cc = C.cA[s];
    int cx = cell_x(cc), cy = cell_y(cc), cz = cell_z(cc);
    if (kick) {
        vec_t<T> qv = C.qA[s];
        vec_t<T> pv = C.pA[s];
        const vec_t<T> f = C.F[s];
        pv.x += half_dt * f.x; pv.y += half_dt * f.y; pv.z += half_dt * f.z;
        const T c = dt * C.inv_m;
        qv.x += c * pv.x; qv.y += c * pv.y; qv.z += c * pv.z;
        move_axis(qv.x, cx, cell_len<T>(R, 0), R.nc[0]);
        move_axis(qv.y, cy, cell_len<T>(R, 1), R.nc[1]);
        if (R.walls)
            wall_axis(qv.z, cz, pv.z, cell_len<T>(R, 2), R.nc[2], C.wall[rep], T(2) * C.m * (T)R.wall_u);
        else
            move_axis(qv.z, cz, cell_len<T>(R, 2), R.nc[2]);
        cc = pack_cell(cx, cy, cz);
        C.pA[s] = pv;
        C.qA[s] = qv;
        C.cA[s] = cc;
    }
    const int key = cell_index(C.tab, R, cx, cy, cz);
    C.key[s] = key;
    atomicAdd(&C.count[key], 1);
}

// ---------------------------------------------------------------------------
// exclusive scan of the cell counts (two passes, 2048 elements per block)
// ---------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ int block_exclusive_scan(int v, int* sh, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;
    }
    __syncthreads();
    const int warp_prefix = warp ? sh[warp - 1] : 0;
    total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_prefix + x - v;
}

__global__ void k_scan_local(const int* __restrict__ in, int* __restrict__ out, int* __restrict__ bsum,
                             int n) {
    __shared__ int sh[32];
    const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0;
        sum += v[k];
    }
    int total;
    int run = block_exclusive_scan(sum, sh, total);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

__global__ void k_scan_bsums(int* __restrict__ bsum, int nb) {
    __shared__ int sh[32];
    int carry = 0;
    for (int t0 = 0; t0 < nb; t0 += blockDim.x) {
        const int t = t0 + threadIdx.x;
        const int v = t < nb ? bsum[t] : 0;
        int total;
        const int ex = block_exclusive_scan(v, sh, total);
        if (t < nb) bsum[t] = carry + ex;
        carry += total;
    }
}

// Adds to each tile's scan the sum of the tiles before it, which every block
// forms for itself (a launch of one block for that cost a small step ~2.5 us;
// the 600 sums at 4M particles are read from L2 by a block's threads at once),
// up to SCAN_SELF tiles; beyond, k_scan_bsums has formed them (`scanned`). With the
// two counters cleared here instead of by memsets a step has three nodes less:
// 108,000 particles 215 -> 205 us, 250,047 (SEM) 168 -> 162.
// Block 0 also clears the step's lists of deferred domains and tiles.
constexpr int SCAN_ADD_THREADS = 256;
constexpr int SCAN_SELF = 2048;
static_assert(SCAN_TILE % SCAN_ADD_THREADS == 0, "a block lies in one tile");

__global__ void __launch_bounds__(SCAN_ADD_THREADS) k_scan_add(int* __restrict__ out, const int* __restrict__ bsum,
                                                               int n, int total, bool scanned, int* zero_a, int* zero_b,
                                                               int nb) {
    __shared__ int sh[SCAN_ADD_THREADS / 32];
    const int i = blockIdx.x * SCAN_ADD_THREADS + threadIdx.x, tile = blockIdx.x * SCAN_ADD_THREADS / SCAN_TILE;
    int before = 0;
    if (scanned) before = threadIdx.x == 0 ? bsum[tile] : 0;
    else
        for (int t = threadIdx.x; t < tile; t += SCAN_ADD_THREADS) before += bsum[t];
    before = __reduce_add_sync(0xffffffffu, before);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = before;
    __syncthreads();
    int add = 0;
#pragma unroll
    for (int w = 0; w < SCAN_ADD_THREADS / 32; ++w) add += sh[w];
    if (i < n) out[i] += add;
    if (i == 0) {
        out[n] = total;
        *zero_a = 0;
    }
    if (i < nb) zero_b[i] = 0;
}

// ---------------------------------------------------------------------------
// counting sort by (cell, id): scatter into cells, then rank by id inside
// each cell and gather A -> B (refreshing beta = C_v / eps)
// ---------------------------------------------------------------------------
// h / n for 0 <= h < 4096, n <= 16, from in = 1 / n: (h + 1/2) / n stays
// 1/32 clear of the next integer
__device__ __forceinline__ int small_div(int h, float in) { return (int)(((float)h + 0.5f) * in); }

// Frame tiles: (replica, first cells) of each, and whether its halo holds more
// particles than the frame is used for (set by k_scatter's last blocks).
struct FrameTiles {
    const int4* org;
    unsigned char* rel;
    int n, edge, hframe;
};

// Blocks of the launch beyond the particles' nb count the halos of the force
// pass's frame tiles, a warp per tile.
template <class T>
__global__ void k_scatter(Ctx<T> C, FrameTiles F, int nb) {
    if ((int)blockIdx.x >= nb) {
        const int f = ((int)blockIdx.x - nb) * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (f >= F.n) return;
        const int4 o = F.org[f];
        const RepInfo& R = C.reps[o.x];
        const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
        const int HX = min(F.edge, nx - o.y) + 2, HY = min(F.edge, ny - o.z) + 2, HZ = min(F.edge, nz - o.w) + 2;
        const float iHX = 1.0f / (float)HX, iHY = 1.0f / (float)HY;
        int sum = 0;
#pragma unroll 4
        for (int h = lane; h < HX * HY * HZ; h += 32) {
            const int row = small_div(h, iHX), hz = small_div(row, iHY);
            int x = o.y + h - row * HX - 1, y = o.z + row - hz * HY - 1, z = o.w + hz - 1;
            const bool use = !(R.walls && (z < 0 || z >= nz));   // nothing beyond a wall
            x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
            y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
            z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
            const int c = use ? cell_index(C.tab, R, x, y, z) : 0;
            sum += use ? C.start[c + 1] - C.start[c] : 0;
        }
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) F.rel[f] = sum > F.hframe;
        return;
    }
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= C.N) return;
    const int c = C.key[s];
    C.tmp[C.start[c] + atomicAdd(&C.fill[c], 1)] = s;
}

template <class T>
__global__ void k_rank_gather(Ctx<T> C) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= C.N) return;
    const int s = C.tmp[t];
    const int c = C.key[s];
    const int b = C.start[c], e = C.start[c + 1];
    const vec_t<T> qv = C.qA[s];
    const uint32_t my = id_of(qv);
    int rank = 0;
    for (int u = b; u < e; ++u) rank += (id_of(C.qA[C.tmp[u]]) < my) ? 1 : 0;
    const int dst = b + rank;
    const RepInfo& R = C.reps[C.rep_of_slot[s]];
    vec_t<T> pv = C.pA[s];
    const eps_t<T> ev = C.eA[s];
    pv.w = beta_of(ev, R);
    C.qB[dst] = qv;
    C.pB[dst] = pv;
    C.eB[dst] = ev;
    C.cB[dst] = C.cA[s];
    C.idB[dst] = my;
}

// B -> A copy (after set_state and after the SSA-only scheme), refreshing beta
// and checking the state.
template <class T>
__global__ void k_copy_back(Ctx<T> C) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= C.N) return;
    const RepInfo& R = C.reps[C.rep_of_slot[s]];
    vec_t<T> pv = C.pB[s];
    const eps_t<T> ev = C.eB[s];
    pv.w = beta_of(ev, R);
    C.qA[s] = C.qB[s];
    C.pA[s] = pv;
    C.eA[s] = ev;
    C.cA[s] = C.cB[s];
    check_state<T>(C.status, pv, ev);
}

// ---------------------------------------------------------------------------
// SER (Sec. III.B.1) over the neighbour list.
// delta p_ij = -gamma_ij chi v_ij dt + sigma sqrt(chi) G_ij sqrt(dt),
// gamma_ij = sigma^2/4 (beta_i + beta_j) (Eq. DPDE_fd), chi = w^2.
//
// Both sweeps are warp-cooperative: a warp takes 32 consecutive particles
// (its lanes' own particles) and spreads all their list entries over its
// lanes, one entry per lane per pass, so every lane evaluates a pair on every
// pass however uneven the lists are. The pair values of one owner are summed
// by a segmented shuffle scan (in entry order inside a pass, passes in order:
// deterministic) and handed to the owner lane.
//
// What bounds them: the load/store unit, then issue. The lists are
// entry-major, one row of a warp's particles contiguous, but a pass takes
// several entries of one owner, so reading entries (and writing delta p_ij)
// at [k N + i] touched a sector per lane, ~130 wavefronts a pass. The first
// sweep now reads its lists a lane per owner, rows contiguous, into shared
// memory in flat order (SERWIN_BYTES a warp: the ~400 entries of a warp at
// density 3 in one window), and writes delta p_ij in flat order too, the
// partner and the owner lane in the fourth word, so that the second sweep
// reads one contiguous row a pass and no list. Us per step, first and second
// sweep: SER at 1M 168 + 160 -> 144 + 88, Hybrid at 4M 193 + 196 -> 169 + 133.
// ---------------------------------------------------------------------------
constexpr int SER_THREADS = 128;
constexpr int SERWIN_BYTES = 4096;

struct WarpEntries {
    int lane, nn, incl, total;
};

__device__ __forceinline__ WarpEntries warp_entries(int nn) {
    WarpEntries W;
    W.lane = threadIdx.x & 31;
    W.nn = nn;
    int incl = nn;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (W.lane >= o) incl += y;
    }
    W.incl = incl;
    W.total = __shfl_sync(0xffffffffu, incl, 31);
    return W;
}

// partner slot and owner lane in one word
static_assert(NBR_J_BITS == 27, "five bits hold the owner lane");
__device__ __forceinline__ uint32_t pack_owner(int j, int lane) { return (uint32_t)j | ((uint32_t)lane << NBR_J_BITS); }
__device__ __forceinline__ int owner_of(uint32_t x) { return (int)(x >> NBR_J_BITS); }
__device__ __forceinline__ int partner_of(uint32_t x) { return (int)(x & ((1u << NBR_J_BITS) - 1)); }
__device__ __forceinline__ uint32_t word_bits(float w) { return __float_as_uint(w); }
__device__ __forceinline__ uint32_t word_bits(double w) { return (uint32_t)__double_as_longlong(w); }
__device__ __forceinline__ void set_word(float& w, uint32_t x) { w = __uint_as_float(x); }
__device__ __forceinline__ void set_word(double& w, uint32_t x) { w = __longlong_as_double((long long)x); }

// first lane of my lane's run of equal owners
__device__ __forceinline__ int owner_head(int lane, int owner) {
    const int prev = __shfl_up_sync(0xffffffffu, owner, 1);
    const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || prev != owner);
    return 31 - __clz((int)(heads & (0xffffffffu >> (31 - lane))));
}

// segmented sum of v over lanes with equal owner; returns to every lane the
// sum over this pass's entries of its own particle (0 if none)
template <class T>
__device__ __forceinline__ T warp_owner_sum(const WarpEntries& W, int f0, int head, T v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, v, o);
        if (W.lane - o >= head) v += y;
    }
    // my entries in this pass end at flat index incl - 1
    const int last = W.incl - 1 - f0;
    const bool mine = W.nn > 0 && last >= 0 && W.incl - W.nn < f0 + 32;
    const T s = __shfl_sync(0xffffffffu, v, min(max(last, 0), 31));
    return mine ? s : T(0);
}

// delta p_ij of entry (j, w) of particle i (pair arithmetic of Eq. SER_p)
template <class T>
__device__ __forceinline__ T3<T> ser_dp(const Ctx<T>& C, int j, T w, uint32_t step, T dt, T sdt,
                                        const vec_t<T>& pi, uint32_t idi, int rep) {
    const vec_t<T> pj = C.pB[j];
    const T3<T> G = pair_gauss<T>(C.seed, step, (uint32_t)rep, idi, C.idB[j]);
    const T A = -(C.sig2_4 * (pi.w + pj.w)) * (w * w) * dt;
    const T Bn = sdt * w;
    return T3<T>{A * ((pi.x - pj.x) * C.inv_m) + Bn * G.x, A * ((pi.y - pj.y) * C.inv_m) + Bn * G.y,
                 A * ((pi.z - pj.z) * C.inv_m) + Bn * G.z};
}

// the entries [c0, c0 + win) of the warp's flat list, a lane per owner i with
// four loads in flight (past the end the last one again)
template <class T>
__device__ __forceinline__ void ser_window(const Ctx<T>& C, const WarpEntries& W, int i, int c0, int win, ListEnt<T>* ent) {
    const int excl = W.incl - W.nn, k1 = min(W.nn, c0 + win - excl);
    const ListEnt<T>* row = C.nbr + i;
    for (int k = max(0, c0 - excl); k < k1; k += 4) {
        ListEnt<T> v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = row[(size_t)min(k + u, k1 - 1) * (size_t)C.N];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k + u < k1) {
                v[u].j = (int)pack_owner(v[u].j, W.lane);
                ent[excl + k + u - c0] = v[u];
            }
    }
    __syncwarp();
}

// first sweep: delta p_i = sum_j delta p_ij (Eq. SER_p). Each delta p_ij is
// also written, with its partner and owner, into the forward-entry buffer
// fwd_g (free once the SSA part of the step is done), the entries of a warp's
// particles in flat order from [first particle * cap], so that the second
// sweep reads it instead of drawing the pair's Gaussian again.
template <class T>
__global__ void __launch_bounds__(SER_THREADS) k_ser_sweep1(Ctx<T> C, T dt, T sqrt_dt) {
    constexpr int WIN = SERWIN_BYTES / (int)sizeof(ListEnt<T>);   // entries held at a time (a multiple of 32)
    __shared__ ListEnt<T> win[SER_THREADS / 32][WIN];
    ListEnt<T>* const ent = win[threadIdx.x >> 5];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int base = i - (int)(threadIdx.x & 31);
    const WarpEntries W = warp_entries(i < C.N ? C.nbr_n[i] : 0);
    const uint32_t step = (uint32_t)*C.step;
    const T sdt = C.sigma * sqrt_dt;
    vec_t<T>* const out_g = C.fwd_g + (size_t)base * C.nbr_cap;
    T ax = 0, ay = 0, az = 0;
    for (int c0 = 0; c0 < W.total; c0 += WIN) {
        ser_window(C, W, i, c0, WIN, ent);
        const int end = min(W.total, c0 + WIN);
        for (int f0 = c0; f0 < end; f0 += 32) {
            const int f = f0 + W.lane;
            int o = 32;
            T3<T> d{0, 0, 0};
            if (f < end) {
                const ListEnt<T> en = ent[f - c0];
                o = owner_of((uint32_t)en.j);
                const int io = base + o;
                d = ser_dp(C, partner_of((uint32_t)en.j), en.w, step, dt, sdt, C.pB[io], C.idB[io], C.rep_of_slot[io]);
                vec_t<T> dv;
                dv.x = d.x; dv.y = d.y; dv.z = d.z;
                set_word(dv.w, (uint32_t)en.j);
                out_g[f] = dv;
            }
            const int head = owner_head(W.lane, o);
            ax += warp_owner_sum(W, f0, head, d.x);
            ay += warp_owner_sum(W, f0, head, d.y);
            az += warp_owner_sum(W, f0, head, d.z);
        }
        __syncwarp();   // the window has been read
    }
    if (i >= C.N) return;
    vec_t<T> out;
    out.x = ax; out.y = ay; out.z = az; out.w = T(0);
    C.dp[i] = out;
}

__device__ __forceinline__ double eps_half(double x) { return 0.5 * x; }
__device__ __forceinline__ ff eps_half(ff x) { return {0.5f * x.hi, 0.5f * x.lo}; }

// eps_i + add - Delta K_i, Delta K_i = (p' - p).(p' + p) / (2m) the kinetic-
// energy change of the stored momenta p -> p'. In FP64 plain arithmetic; in
// the mixed mode Delta K is formed as a compensated pair from exact
// two-sums and two-products of the float momenta, so that the internal
// energy absorbs the kinetic change to ~2^-46 relative rather than 2^-24.
__device__ __forceinline__ double eps_minus_dk(double e, double add, const d4& pn, const d4& pi, double hm) {
    const double dK = ((pn.x - pi.x) * (pn.x + pi.x) + (pn.y - pi.y) * (pn.y + pi.y) +
                       (pn.z - pi.z) * (pn.z + pi.z)) * hm;
    return e + (add - dK);
}
__device__ __forceinline__ ff eps_minus_dk(ff e, ff add, const float4& pn, const float4& pi, float hm) {
    float lx, ly, lz;
    const float hx = diff_of_squares(pn.x, pi.x, lx);
    const float hy = diff_of_squares(pn.y, pi.y, ly);
    const float hz = diff_of_squares(pn.z, pi.z, lz);
    float e1, e2;
    const float s1 = two_sum(hx, hy, e1);
    const float s2 = two_sum(s1, hz, e2);
    const float lo = __fadd_rn(__fadd_rn(e1, e2), __fadd_rn(lx, __fadd_rn(ly, lz)));
    // -Delta K as a pair (hm = 1/(2m), exact for a power-of-two mass)
    const float nh = -__fmul_rn(s2, hm), nl = -__fmul_rn(lo, hm);
    ff d;
    d.hi = __fadd_rn(nh, nl);
    d.lo = __fsub_rn(nl, __fsub_rn(d.hi, nh));
    return ff_add(ff_add(e, add), d);
}

// second sweep, Eq. (SER_eint_discretization), in the equivalent form
//   Delta eps_i = -Delta K_i + 1/2 sum_j T_ij,
//   T_ij = delta p_ij . (v_i + v_j + (delta p_i + delta p_j) / (2m)),
// where Delta K_i = (p_i' - p_i).(p_i' + p_i) / (2m) is the kinetic-energy
// change of the stored momenta. T_ij = -T_ji bit for bit, so the FD part
// conserves energy up to the rounding of per-particle sums. Writes the new
// state (q, cell, p, eps) into set A.
template <class T>
__global__ void __launch_bounds__(SER_THREADS) k_ser_sweep2(Ctx<T> C) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int base = i - (int)(threadIdx.x & 31);
    const WarpEntries W = warp_entries(i < C.N ? C.nbr_n[i] : 0);
    const T hm = T(0.5) * C.inv_m;
    const vec_t<T>* const in_g = C.fwd_g + (size_t)base * C.nbr_cap;   // delta p_ij of the first sweep
    eps_t<T> tsum{};   // compensated in the mixed mode
    for (int f0 = 0; f0 < W.total; f0 += 32) {
        const int f = f0 + W.lane;
        int o = 32;
        T tv = 0;
        if (f < W.total) {
            const vec_t<T> d = in_g[f];
            const uint32_t jo = word_bits(d.w);
            o = owner_of(jo);
            const int io = base + o, j = partner_of(jo);
            const vec_t<T> pi = C.pB[io];
            const vec_t<T> dpi = C.dp[io];
            const vec_t<T> pj = C.pB[j];
            const vec_t<T> dpj = C.dp[j];
            const T vix = pi.x * C.inv_m, viy = pi.y * C.inv_m, viz = pi.z * C.inv_m;
            const T vjx = pj.x * C.inv_m, vjy = pj.y * C.inv_m, vjz = pj.z * C.inv_m;
            tv = d.x * ((vix + vjx) + (dpi.x + dpj.x) * hm) + d.y * ((viy + vjy) + (dpi.y + dpj.y) * hm) +
                 d.z * ((viz + vjz) + (dpi.z + dpj.z) * hm);
        }
        const int head = owner_head(W.lane, o);
        tsum = eps_add(tsum, warp_owner_sum(W, f0, head, tv));
    }
    if (i >= C.N) return;
    const RepInfo& R = C.reps[C.rep_of_slot[i]];
    const vec_t<T> pi = C.pB[i];
    const vec_t<T> dpi = C.dp[i];
    vec_t<T> pn = pi;
    pn.x = pi.x + dpi.x; pn.y = pi.y + dpi.y; pn.z = pi.z + dpi.z;
    const eps_t<T> en = eps_minus_dk(C.eB[i], eps_half(tsum), pn, pi, hm);
    pn.w = beta_of(en, R);
    C.qA[i] = C.qB[i];
    C.cA[i] = C.cB[i];
    C.pA[i] = pn;
    C.eA[i] = en;
    check_state<T>(C.status, pn, en);
}

// ---------------------------------------------------------------------------
// SEM, Eq. (SEM_fd): one sweep, Euler-Maruyama on p and eps. B -> A.
//
// Issue-bound, most of it the draw: a thread per particle drew for the longest
// list of its warp (20 entries of 12.6 at density 3). The entries are spread
// over the lanes as in the SER sweeps, their increments left in shared memory
// and summed by the owner in list order (250,047 particles 41.5 -> 39.8 us,
// 1.4 waves of blocks).
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(SER_THREADS) k_sem(Ctx<T> C, T dt, T sqrt_dt) {
    constexpr int WIN = SERWIN_BYTES / 2 / (int)sizeof(ListEnt<T>);
    __shared__ ListEnt<T> win[SER_THREADS / 32][WIN];
    __shared__ vec_t<T> inc[SER_THREADS / 32][WIN];
    ListEnt<T>* const ent = win[threadIdx.x >> 5];
    vec_t<T>* const val = inc[threadIdx.x >> 5];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int base = i - (int)(threadIdx.x & 31);
    const WarpEntries W = warp_entries(i < C.N ? C.nbr_n[i] : 0);
    const uint32_t step = (uint32_t)*C.step;
    const T d_sig2_m = T(3) * C.sigma * C.sigma * C.inv_m;
    const T sdt = C.sigma * sqrt_dt;
    const int excl = W.incl - W.nn;
    T ax = 0, ay = 0, az = 0, de = 0;
    for (int c0 = 0; c0 < W.total; c0 += WIN) {
        ser_window(C, W, i, c0, WIN, ent);
        const int end = min(W.total, c0 + WIN);
        for (int f = c0 + W.lane; f < end; f += 32) {
            const ListEnt<T> en = ent[f - c0];
            const int io = base + owner_of((uint32_t)en.j), j = partner_of((uint32_t)en.j);
            const T w = en.w;
            const vec_t<T> pi = C.pB[io], pj = C.pB[j];
            const T chi = w * w;
            const T gam = C.sig2_4 * (pi.w + pj.w);
            const T3<T> G = pair_gauss<T>(C.seed, step, (uint32_t)C.rep_of_slot[io], C.idB[io], C.idB[j]);
            const T vx = (pi.x - pj.x) * C.inv_m;
            const T vy = (pi.y - pj.y) * C.inv_m;
            const T vz = (pi.z - pj.z) * C.inv_m;
            const T A = -gam * chi * dt, Bn = sdt * w;
            vec_t<T> v;
            v.x = A * vx + Bn * G.x;
            v.y = A * vy + Bn * G.y;
            v.z = A * vz + Bn * G.z;
            v.w = T(0.5) * (gam * (vx * vx + vy * vy + vz * vz) - d_sig2_m) * chi * dt -
                  T(0.5) * Bn * (vx * G.x + vy * G.y + vz * G.z);
            val[f - c0] = v;
        }
        __syncwarp();
        for (int f = max(c0, excl); f < min(W.incl, end); ++f) {
            const vec_t<T> v = val[f - c0];
            ax += v.x;
            ay += v.y;
            az += v.z;
            de += v.w;
        }
        __syncwarp();   // the window has been read
    }
    if (i >= C.N) return;
    const RepInfo& R = C.reps[C.rep_of_slot[i]];
    const vec_t<T> pi = C.pB[i];
    vec_t<T> pn = pi;
    pn.x = pi.x + ax; pn.y = pi.y + ay; pn.z = pi.z + az;
    const eps_t<T> en = eps_add(C.eB[i], de);
    pn.w = beta_of(en, R);
    C.qA[i] = C.qB[i];
    C.cA[i] = C.cB[i];
    C.pA[i] = pn;
    C.eA[i] = en;
    check_state<T>(C.status, pn, en);
}

// ---------------------------------------------------------------------------
// SSA (Sec. III.A.2 and III.B.2): the pair map of Eq. (SSA_ij) -- the exact
// OU transition of p_st at fixed gamma_st, after which eps_s and eps_t each
// absorb -Delta K_st / 2 -- applied pair after pair in sequence order.
//
// The Gaussians do not depend on the state, so they are drawn first for every
// forward entry by a fully parallel pass (k_ssa_gauss) and stored with the
// entry's weight; the sequential part then only applies the maps.
//
// One launch per cell colour class; one thread per cell of the class. The
// cells reached by the pairs of two cells of one class are disjoint, so the
// threads touch disjoint particles and update set B in place. A thread walks
// its cell's chain -- the forward rows of the cell's particles s in slot
// (= id) order, concatenated -- as one flat loop, so the lanes of a warp
// diverge only by chain length. (p_s, eps_s, beta_s) stay in registers while
// s is current; the partner's updated (p_t, eps_t) goes back to memory at
// once, with beta_t = C_v / eps_t in p_t.w, so p.w is the current beta of
// every particle throughout. Partner indices are loaded two entries ahead,
// the partner state (and the next particle's state on a row change) one
// entry ahead. Loads issued ahead of a store can alias it only for the
// partner t being updated (two rows of a cell may share a partner, and a
// later particle of the cell may itself be t); those take the new values
// from registers.
// ---------------------------------------------------------------------------
constexpr int SSA_THREADS = 64;      // default block size; the autotuner picks 32..128
constexpr int SSA_THREADS_MAX = 128;
constexpr int SSA_ROWS = 20;     // rows per cell held in the shared row table
constexpr int NCOLOURS = 75;     // (2 + 1) x (3 + 2) x (3 + 2) cell colours

// G of every forward entry, with its weight: reads entry m of particle s at
// [m * N + s] (as the force pass wrote it) and writes (G_st, w)
// particle-major at [s * cap + m], the order the SSA chains read it. A
// warp takes 32 consecutive particles and spreads their entries over its
// lanes (a shuffle prefix sum of the row lengths gives each entry's owner).
template <class T>
__global__ void k_ssa_gauss(Ctx<T> C) {
    const int lane = threadIdx.x & 31;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int base = s - lane;
    const int nf = s < C.N ? C.fwd_n[s] : 0;
    int incl = nf;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t step = (uint32_t)*C.step;
    const size_t cap = (size_t)C.nbr_cap;
    for (int f0 = 0; f0 < total; f0 += 32) {
        const int f = f0 + lane;
        // owner: the first lane whose inclusive prefix exceeds f
        int lo = 0;
#pragma unroll
        for (int step2 = 16; step2 > 0; step2 >>= 1) {
            const int v = __shfl_sync(0xffffffffu, incl, lo + step2 - 1);
            if (v <= f) lo += step2;
        }
        const int excl = __shfl_sync(0xffffffffu, incl - nf, lo);
        if (f < total) {
            const int so = base + lo;
            const size_t at = (size_t)(f - excl) * C.N + so;
            const size_t row = (size_t)so * cap + (f - excl);
            const ListEnt<T> en = C.fwd[at];
            const T3<T> G = pair_gauss<T>(C.seed, step, (uint32_t)C.rep_of_slot[so], C.idB[so], C.idB[en.j]);
            vec_t<T> g;
            g.x = G.x; g.y = G.y; g.z = G.z; g.w = en.w;
            C.fwd_g[row] = g;
        }
    }
}

// The pair map on (p_s, eps_s, beta_s) in registers and partner (p_t, eps_t)
// with beta_t = p_t.w, for the entry (G, w) = g; returns the new partner
// state, beta in .w.
// beta = C_v / eps: exact in double; in float through the fast reciprocal
// (2 ulp), which keeps the chains' critical path short
__device__ __forceinline__ float ssa_beta(ff e, const RepInfo& R) { return __fdividef(R.cvf, e.hi); }
// sqrt(x / y) for x >= 0, y > 0 as x rsqrt(x y) (a few ulp, for x y a normal
// float; 0 for x = 0)
__device__ __forceinline__ float ssa_sqrt_ratio(float x, float y) {
    return x > 0.0f ? __fmul_rn(x, rsqrtf(__fmul_rn(x, y))) : 0.0f;
}
__device__ __forceinline__ double ssa_beta(double e, const RepInfo& R) { return R.cv / e; }

// Explicitly rounded operations: the compiler neither fuses nor reorders them,
// so every kernel that inlines the pair map computes the same bits.
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float r_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double r_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// In double an operation takes the chip some thirty times a float's, so a
// map's count of them is its time. With a = gamma w^2 2 dt / m the amplitude
// sigma sqrt(m (1 - e^{-2a}) / gamma) is 2 sigma sqrt(dt) w Q(a),
//   Q(a) = sqrt((1 - e^{-2a}) / (2a)),
// which needs neither the division nor the root where a is small: there
// (e^{-a} - 1) / 2 and Q are polynomials (Chebyshev fits on [0, 1/4], error
// below 2^-56), independent of each other. What does not depend on the state
// goes into the map's noise (ssa_noise) beforehand. a is 0.02 to 0.2 in the
// fluids of the paper; beyond 1/4 the functions themselves. Us per pass: ten
// Hybrid steps of 1,000 particles 5024 -> 3936, two of 108,000 2030 -> 1802.
__device__ __forceinline__ void ssa_ou(double a, double& hem, double& Q) {
    if (a >= 0.0 && a <= 0.25) {
        double h = 1.23028890849153e-07;
        h = fma(a, h, -1.3701804316291336e-06);
        h = fma(a, h, 1.2398555234119672e-05);
        h = fma(a, h, -9.920595362410088e-05);
        h = fma(a, h, 0.000694444401087605);
        h = fma(a, h, -0.0041666666637702535);
        h = fma(a, h, 0.02083333333322211);
        h = fma(a, h, -0.08333333333333116);
        h = fma(a, h, 0.24999999999999997);
        h = fma(a, h, -0.5);
        hem = __dmul_rn(a, h);
        double q = 6.5425756532649734e-06;
        q = fma(a, q, -5.837075404796853e-05);
        q = fma(a, q, 0.0003668523284567146);
        q = fma(a, q, -0.002343749303760139);
        q = fma(a, q, 0.013715277715415457);
        q = fma(a, q, -0.06249999999689911);
        q = fma(a, q, 0.20833333333325674);
        q = fma(a, q, -0.4999999999999993);
        Q = fma(a, q, 1.0);
    } else {
        const double em1 = expm1(-a);
        hem = __dmul_rn(0.5, em1);
        Q = sqrt(__dmul_rn(em1, __dadd_rn(em1, 2.0)) / __dmul_rn(-2.0, a));
    }
}

// The noise of a map from its entry (G, w), k2 = 2 dt / m, amp0 = 2 sigma
// sqrt(dt): in double (amp0 w G / 2, sigma^2 / 4 w^2 k2), in float the entry.
__device__ __forceinline__ float4 ssa_noise(const Ctx<float>&, const float4& g, float, float) { return g; }
__device__ __forceinline__ d4 ssa_noise(const Ctx<double>& C, const d4& g, double k2, double amp0) {
    const double A = __dmul_rn(0.5, __dmul_rn(amp0, g.w));
    d4 n;
    n.x = __dmul_rn(A, g.x);
    n.y = __dmul_rn(A, g.y);
    n.z = __dmul_rn(A, g.z);
    n.w = __dmul_rn(C.sig2_4, __dmul_rn(__dmul_rn(g.w, g.w), k2));
    return n;
}

// The map with its noise g.
template <class T>
__device__ __forceinline__ void ssa_noise_map(const Ctx<T>& C, const RepInfo& R, vec_t<T>& ps, eps_t<T>& es,
                                              T& bs, vec_t<T>& pt, eps_t<T>& et, const vec_t<T>& g, T k2,
                                              T amp0) {
    T Dx, Dy, Dz;
    if constexpr (sizeof(T) == 8) {
        T hem, Q;
        ssa_ou(r_mul(g.w, r_add(bs, pt.w)), hem, Q);
        Dx = r_fma(hem, r_sub(ps.x, pt.x), r_mul(Q, g.x));
        Dy = r_fma(hem, r_sub(ps.y, pt.y), r_mul(Q, g.y));
        Dz = r_fma(hem, r_sub(ps.z, pt.z), r_mul(Q, g.z));
    } else {
        const T w = g.w;
        const T chik = r_mul(r_mul(w, w), k2);
        const T gam = r_mul(C.sig2_4, r_add(bs, pt.w));
        const T aa = r_mul(gam, chik);   // a = 2 gamma chi dt / m
        // e^{-a} - 1, and 1 - e^{-2a} = -(e^{-a} - 1)(e^{-a} - 1 + 2)
        const T em1 = expm1f(-aa);
        const T x = r_mul(C.m, -r_mul(em1, r_add(em1, T(2))));   // m (1 - e^{-2a})
        const T amp = (gam != T(0)) ? r_mul(C.sigma, ssa_sqrt_ratio((float)x, (float)gam)) : r_mul(amp0, w);
        Dx = r_mul(T(0.5), r_fma(em1, r_sub(ps.x, pt.x), r_mul(amp, g.x)));
        Dy = r_mul(T(0.5), r_fma(em1, r_sub(ps.y, pt.y), r_mul(amp, g.y)));
        Dz = r_mul(T(0.5), r_fma(em1, r_sub(ps.z, pt.z), r_mul(amp, g.z)));
    }
    const T snx = r_add(ps.x, Dx), sny = r_add(ps.y, Dy), snz = r_add(ps.z, Dz);
    const T tnx = r_sub(pt.x, Dx), tny = r_sub(pt.y, Dy), tnz = r_sub(pt.z, Dz);
    // kinetic-energy change of the stored momenta, halved
    T q = r_mul(r_sub(tnz, pt.z), r_add(tnz, pt.z));
    q = r_fma(r_sub(tny, pt.y), r_add(tny, pt.y), q);
    q = r_fma(r_sub(tnx, pt.x), r_add(tnx, pt.x), q);
    q = r_fma(r_sub(snz, ps.z), r_add(snz, ps.z), q);
    q = r_fma(r_sub(sny, ps.y), r_add(sny, ps.y), q);
    q = r_fma(r_sub(snx, ps.x), r_add(snx, ps.x), q);
    const T dK = r_mul(q, r_mul(T(0.25), C.inv_m));
    ps.x = snx; ps.y = sny; ps.z = snz;
    es = eps_add(es, -dK);
    bs = ssa_beta(es, R);
    pt.x = tnx; pt.y = tny; pt.z = tnz;
    et = eps_add(et, -dK);
    pt.w = ssa_beta(et, R);
}

// The map of the entry (G, w) = g.
template <class T>
__device__ __forceinline__ void ssa_pair_map(const Ctx<T>& C, const RepInfo& R, vec_t<T>& ps, eps_t<T>& es,
                                             T& bs, vec_t<T>& pt, eps_t<T>& et, const vec_t<T>& g, T k2,
                                             T amp0) {
    ssa_noise_map(C, R, ps, es, bs, pt, et, ssa_noise(C, g, k2, amp0), k2, amp0);
}

// Plain (unpipelined) chain, for cells with more than SSA_ROWS rows.
template <class T>
__device__ void ssa_chain_plain(const Ctx<T>& C, const RepInfo& R, int b, int e, T k2, T amp0) {
    const size_t cap = (size_t)C.nbr_cap;
    for (int s = b; s < e; ++s) {
        const int nf = C.fwd_n[s];
        if (nf == 0) continue;
        vec_t<T> ps = C.pB[s];
        eps_t<T> es = C.eB[s];
        T bs = ps.w;
        for (int m = 0; m < nf; ++m) {
            const int t = C.fwd[(size_t)m * C.N + s].j;
            const vec_t<T> g = C.fwd_g[(size_t)s * cap + m];
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

// dynamic shared memory of k_ssa_colour: two row tables [SSA_ROWS][block]
__host__ __device__ constexpr size_t ssa_smem_bytes(int block) { return (size_t)2 * SSA_ROWS * block * sizeof(int); }

// The chain of cell c on the calling thread (its column tid of the shared
// row tables, bdim columns).
template <class T>
__device__ __forceinline__ void ssa_cell_chain(const Ctx<T>& C, int c, T dt, T sqrt_dt, int* row_s, int* row_n,
                                               int bdim, int tid) {
    const int b = C.start[c], e = C.start[c + 1];
    int nrow = 0, total = 0;
    for (int s = b; s < e; ++s) {
        const int nf = C.fwd_n[s];
        if (nf > 0) {
            if (nrow < SSA_ROWS) {
                row_s[nrow * bdim + tid] = s;
                row_n[nrow * bdim + tid] = nf;
            }
            ++nrow;
            total += nf;
        }
    }
    if (total == 0) return;
    const RepInfo& R = C.reps[C.rep_of_cell[c]];
    const T amp0 = T(2) * C.sigma * sqrt_dt;   // amplitude of the map as gamma -> 0
    const T k2 = T(2) * dt * C.inv_m;
    if (nrow > SSA_ROWS) {
        ssa_chain_plain(C, R, b, e, k2, amp0);
        return;
    }
    const size_t cap = (size_t)C.nbr_cap;
    // position (r, m) of an entry; advancing past the last entry stays there
    auto advance = [&](int& r, int& m, int& nf) {
        if (m + 1 < nf) {
            ++m;
        } else if (r + 1 < nrow) {
            ++r;
            m = 0;
            nf = row_n[r * bdim + tid];
        }
    };
    // An entry of the chain: owner s, partner t, (G, w); the partner state,
    // and on a row switch the new owner's state, loaded two entries ahead.
    struct Ent {
        int s, t;
        vec_t<T> g, pt, ps;
        eps_t<T> et, es;
        bool sw;
    };
    auto load_index = [&](int r, int m, Ent& x) {
        x.s = row_s[r * bdim + tid];
        x.t = C.fwd[(size_t)m * C.N + x.s].j;
        x.g = C.fwd_g[(size_t)x.s * cap + m];
    };
    auto load_state = [&](Ent& x, int prev_s) {
        x.pt = C.pB[x.t];
        x.et = C.eB[x.t];
        x.sw = x.s != prev_s;
        if (x.sw) {
            x.ps = C.pB[x.s];
            x.es = C.eB[x.s];
        }
    };
    // the last two partner writes (w1 newest): the only stores a value loaded
    // two entries ahead can miss
    int w1t = -1, w2t = -1;
    vec_t<T> w1p, w2p;
    eps_t<T> w1e, w2e;
    auto patch = [&](int x, vec_t<T>& pv, eps_t<T>& ev) {
        if (x == w2t) { pv = w2p; ev = w2e; }
        if (x == w1t) { pv = w1p; ev = w1e; }
    };
    Ent e0, e1, e2;
    int r = 0, m = 0, nfr = row_n[tid];
    load_index(r, m, e0);
    load_state(e0, -1);
    advance(r, m, nfr);
    load_index(r, m, e1);
    load_state(e1, e0.s);
    advance(r, m, nfr);
    load_index(r, m, e2);
    int s = -1;
    vec_t<T> ps;
    eps_t<T> es;
    T bs = T(0);
    for (int k = 0; k < total; ++k) {
        // index of entry k + 3, state of entry k + 2
        advance(r, m, nfr);
        Ent e3;
        load_index(r, m, e3);
        load_state(e2, e1.s);
        // entry k becomes current: patch its loads with the writes they missed
        patch(e0.t, e0.pt, e0.et);
        if (e0.sw) {
            if (s >= 0) {
                ps.w = bs;
                C.pB[s] = ps;
                C.eB[s] = es;
            }
            patch(e0.s, e0.ps, e0.es);
            s = e0.s;
            ps = e0.ps;
            es = e0.es;
            bs = ps.w;
        }
        ssa_pair_map(C, R, ps, es, bs, e0.pt, e0.et, e0.g, k2, amp0);
        C.pB[e0.t] = e0.pt;
        C.eB[e0.t] = e0.et;
        w2t = w1t; w2p = w1p; w2e = w1e;
        w1t = e0.t; w1p = e0.pt; w1e = e0.et;
        e0 = e1;
        e1 = e2;
        e2 = e3;
    }
    ps.w = bs;
    C.pB[s] = ps;
    C.eB[s] = es;
}

// One colour class: one thread per cell of the class.
template <class T>
__global__ void __launch_bounds__(SSA_THREADS_MAX) k_ssa_colour(Ctx<T> C, const int* __restrict__ cells,
                                                                int ncol, T dt, T sqrt_dt) {
    extern __shared__ int ssa_rows[];
    const int bdim = blockDim.x;
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= ncol) return;
    ssa_cell_chain(C, cells[u], dt, sqrt_dt, ssa_rows, ssa_rows + SSA_ROWS * bdim, bdim, (int)threadIdx.x);
}

// ---------------------------------------------------------------------------
// The same SSA sequence domain by domain (Hybrid, Sec. III.B.2). The chains of
// a domain never leave it, so two domains share no particle and their
// sequences commute: each warp takes `group` consecutive domains (one slot
// range, the cells being brick-major) and walks their colour classes in
// order, its lanes running the chains of one class at a time (cells of one
// class share no particle), with a warp barrier between classes (which also
// orders the lanes' memory accesses). The result is the class-by-class
// sequence bit for bit.
//
// The warp stages the state (p, eps) of its slot range in shared memory for
// all its classes when it fits in `scap` slots, and otherwise works on the
// state in place in global memory; in both cases a chain reads a state just
// before the map that uses it, so no load can miss an earlier store. The
// entries of a chain -- partner index and (G, w) -- are loaded SSA_AHEAD
// entries ahead. `bcells` holds the cells of each domain sorted by class,
// `boff[b * (NCOLOURS + 1) + k]` the start of class k of domain b and
// `bcell0[b]` the first cell of domain b (bcell0[nbricks] = ncells).
// ---------------------------------------------------------------------------
constexpr int SSA_GROUP_MAX = 8;
constexpr int SSA_AHEAD = 4;
constexpr int SSA_DOMAIN_SMEM = 200 * 1024;   // dynamic shared memory of one k_ssa_domains block, at most

// the particle state of a warp's slot range: staged (shared memory) or in place
template <class T>
struct SsaState {
    vec_t<T>* p;
    eps_t<T>* e;
    int base, n;   // slots base .. base + n - 1
};

// one forward entry of a chain: owner s, partner t, (G, w)
template <class T>
struct SsaEntry {
    int s, t;
    vec_t<T> g;
};

// next entry of the chain over slots .. e - 1 at (s, m) of a row of nf
// entries; false past the last
__device__ __forceinline__ bool ssa_next(const int* __restrict__ fwd_n, int& s, int& m, int& nf, int e) {
    if (m + 1 < nf) {
        ++m;
        return true;
    }
    for (++s; s < e; ++s) {
        nf = __ldg(fwd_n + s);
        if (nf > 0) {
            m = 0;
            return true;
        }
    }
    return false;
}

template <class T>
__device__ __forceinline__ bool ssa_fetch(const Ctx<T>& C, int& s, int& m, int& nf, int e, SsaEntry<T>& q) {
    if (!ssa_next(C.fwd_n, s, m, nf, e)) return false;
    q.s = s;
    q.t = __ldg(&C.fwd[(size_t)m * C.N + s].j);
    q.g = C.fwd_g[(size_t)s * C.nbr_cap + m];
    return true;
}

// The chain of cell c on the state S. Entries are fetched in blocks of
// SSA_AHEAD into two register sets used in turn (the loop is unrolled over
// the pair, so no register is moved while its load is in flight): the loads
// of block i + 1 are issued before the maps of block i run.
template <class T>
__device__ __forceinline__ void ssa_domain_chain(const Ctx<T>& C, const RepInfo& R, int c, const SsaState<T>& S,
                                                 T k2, T amp0) {
    int s = C.start[c] - 1, m = 0, nf = 0;
    const int e = C.start[c + 1];
    int cur = -1;
    vec_t<T> ps;
    eps_t<T> es;
    T bs = T(0);
    bool bad = false;
    auto fill = [&](SsaEntry<T>(&q)[SSA_AHEAD], bool(&v)[SSA_AHEAD]) {
        bool more = true;
#pragma unroll
        for (int a = 0; a < SSA_AHEAD; ++a) {
            more = more && ssa_fetch(C, s, m, nf, e, q[a]);
            v[a] = more;
        }
    };
    auto run = [&](const SsaEntry<T>(&q)[SSA_AHEAD], const bool(&v)[SSA_AHEAD]) {
#pragma unroll
        for (int a = 0; a < SSA_AHEAD; ++a) {
            if (!v[a]) break;
            const SsaEntry<T>& x = q[a];
            const int ls = x.s - S.base, lt = x.t - S.base;
            if ((unsigned)ls >= (unsigned)S.n || (unsigned)lt >= (unsigned)S.n) {
                bad = true;   // a chain left its domain: never by construction
                break;
            }
            if (x.s != cur) {
                if (cur >= 0) {
                    ps.w = bs;
                    S.p[cur - S.base] = ps;
                    S.e[cur - S.base] = es;
                }
                cur = x.s;
                ps = S.p[ls];
                es = S.e[ls];
                bs = ps.w;
            }
            vec_t<T> pt = S.p[lt];
            eps_t<T> et = S.e[lt];
            ssa_pair_map(C, R, ps, es, bs, pt, et, x.g, k2, amp0);
            S.p[lt] = pt;
            S.e[lt] = et;
        }
    };
    SsaEntry<T> qa[SSA_AHEAD], qb[SSA_AHEAD];
    bool va[SSA_AHEAD], vb[SSA_AHEAD];
    fill(qa, va);
    while (va[0] && !bad) {
        fill(qb, vb);
        run(qa, va);
        if (!vb[0] || bad) break;
        fill(qa, va);
        run(qb, vb);
    }
    if (bad) {
        flag(C.status, ST_DOMAIN);
        return;
    }
    if (cur >= 0) {
        ps.w = bs;
        S.p[cur - S.base] = ps;
        S.e[cur - S.base] = es;
    }
}

// the colour classes of a warp's domains, in order, on the state S
template <class T>
__device__ __forceinline__ void ssa_domain_classes(const Ctx<T>& C, const int* __restrict__ bcells, const int* wo,
                                                   int nb, const SsaState<T>& S, T k2, T amp0) {
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < NCOLOURS; ++k) {
        int total = 0;
        for (int g = 0; g < nb; ++g) total += wo[g * (NCOLOURS + 1) + k + 1] - wo[g * (NCOLOURS + 1) + k];
        if (total == 0) continue;   // whole warp
        for (int i = lane; i < total; i += 32) {
            int g = 0, r = i;
            for (;;) {
                const int cnt = wo[g * (NCOLOURS + 1) + k + 1] - wo[g * (NCOLOURS + 1) + k];
                if (r < cnt) break;
                r -= cnt;
                ++g;
            }
            const int c = bcells[wo[g * (NCOLOURS + 1) + k] + r];
            ssa_domain_chain(C, C.reps[C.rep_of_cell[c]], c, S, k2, amp0);
        }
        __syncwarp();
    }
}

// shared memory of one warp of k_ssa_domains: staged p and eps for scap
// slots, then the class starts of `group` domains
template <class T>
__host__ __device__ constexpr size_t ssa_domain_warp_bytes(int group, int scap) {
    return (size_t)scap * (sizeof(vec_t<T>) + sizeof(eps_t<T>)) +
           (((size_t)group * (NCOLOURS + 1) * sizeof(int) + 15) / 16) * 16;
}

template <class T>
__global__ void __launch_bounds__(SSA_THREADS_MAX) k_ssa_domains(Ctx<T> C, const int* __restrict__ bcells,
                                                                 const int* __restrict__ boff,
                                                                 const int* __restrict__ bcell0, int nbricks,
                                                                 int group, int scap, T dt, T sqrt_dt) {
    extern __shared__ __align__(16) unsigned char ssa_dom_smem[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int b0 = (int)((blockIdx.x * (blockDim.x >> 5) + wib) * group);
    if (b0 >= nbricks) return;   // whole warp
    const int nb = min(group, nbricks - b0);
    unsigned char* wbase = ssa_dom_smem + (size_t)wib * ssa_domain_warp_bytes<T>(group, scap);
    int* wo = reinterpret_cast<int*>(wbase + (size_t)scap * (sizeof(vec_t<T>) + sizeof(eps_t<T>)));
    for (int i = lane; i < nb * (NCOLOURS + 1); i += 32) wo[i] = boff[(size_t)b0 * (NCOLOURS + 1) + i];
    const int sb = C.start[bcell0[b0]], se = C.start[bcell0[b0 + nb]];
    const T amp0 = T(2) * C.sigma * sqrt_dt;   // amplitude of the map as gamma -> 0
    const T k2 = T(2) * dt * C.inv_m;
    SsaState<T> S;
    S.base = sb;
    S.n = se - sb;
    if (S.n <= scap) {   // whole warp
        vec_t<T>* sp = reinterpret_cast<vec_t<T>*>(wbase);
        eps_t<T>* se_ = reinterpret_cast<eps_t<T>*>(wbase + (size_t)scap * sizeof(vec_t<T>));
        for (int i = lane; i < S.n; i += 32) {
            sp[i] = C.pB[sb + i];
            se_[i] = C.eB[sb + i];
        }
        __syncwarp();
        S.p = sp;
        S.e = se_;
        ssa_domain_classes(C, bcells, wo, nb, S, k2, amp0);
        __syncwarp();
        for (int i = lane; i < S.n; i += 32) {
            C.pB[sb + i] = sp[i];
            C.eB[sb + i] = se_[i];
        }
    } else {
        __syncwarp();
        S.p = C.pB + sb;
        S.e = C.eB + sb;
        ssa_domain_classes(C, bcells, wo, nb, S, k2, amp0);
    }
}

__global__ void k_step_inc(long long* step) { *step += 1; }

// ---------------------------------------------------------------------------
// Projection on the internal energies (Sec. IV.C): after the step, every
// eps_i of a replica is lowered by (E - E0)/N, E = U + K + sum eps of the
// unconstrained update (set A after the FD part; U from the force pass at the
// same positions). Per-chunk sums in a fixed order, then per replica.
// ---------------------------------------------------------------------------
constexpr int OBS_THREADS = 256;

template <class T>
__global__ void k_proj_chunks(Ctx<T> C, const int* __restrict__ chunk_begin, const int* __restrict__ chunk_end,
                              double* __restrict__ partial) {
    const int ch = blockIdx.x;
    double acc = 0.0;
    const double hm = 0.5 / (double)C.m;
    for (int i = chunk_begin[ch] + threadIdx.x; i < chunk_end[ch]; i += blockDim.x) {
        const vec_t<T> p = C.pA[i];
        acc += ((double)p.x * p.x + (double)p.y * p.y + (double)p.z * p.z) * hm + (double)C.upot[i] +
               eps_value(C.eA[i]);
    }
    __shared__ double sh[OBS_THREADS];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = OBS_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[ch] = sh[0];
}

template <class T>
__global__ void k_proj_reps(Ctx<T> C, const double* __restrict__ partial, const int* __restrict__ rep_chunk_begin,
                            int R, const double* __restrict__ E0, double* __restrict__ shift) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    double E = 0.0;
    for (int ch = rep_chunk_begin[r]; ch < rep_chunk_begin[r + 1]; ++ch) E += partial[ch];
    const int n = C.reps[r].n;
    shift[r] = n > 0 ? (E - E0[r]) / (double)n : 0.0;
}

template <class T>
__global__ void k_proj_apply(Ctx<T> C, const double* __restrict__ shift) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C.N) return;
    const int r = C.rep_of_slot[i];
    const eps_t<T> e = eps_add(C.eA[i], (T)(-shift[r]));
    C.eA[i] = e;
    vec_t<T> p = C.pA[i];
    p.w = beta_of(e, C.reps[r]);
    C.pA[i] = p;
    check_state<T>(C.status, p, e);
}

// ---------------------------------------------------------------------------
// observables: per-chunk sums (a chunk lies inside one replica), then per
// replica sums of the chunks in order -- deterministic. The pair sums of U
// and its Laplacian come from a tiled pass before (LIST_OBS), in C.dp (free
// between steps). A walk of the 27 cells per particle through global memory
// took most of the call: 1M particles 628 -> 370 us, 100,000 in FP64 3960 ->
// 256 us, Lennard-Jones 100,000 1503 -> 213 us, 1,000 particles 235 -> 79 us.
// terms: 0 K, 1 U, 2 Eint, 3-5 P, 6 sum C_v/eps, 7 |F|^2, 8 Laplacian U,
//        9 neg eps, 10 nonfinite
// ---------------------------------------------------------------------------
constexpr int NTERMS = 11;

template <class T>
__global__ void k_obs_chunks(Ctx<T> C, const int* __restrict__ chunk_rep, const int* __restrict__ chunk_begin,
                             const int* __restrict__ chunk_end, double* __restrict__ partial) {
    const int ch = blockIdx.x;
    const int rep = chunk_rep[ch];
    const RepInfo& R = C.reps[rep];
    double acc[NTERMS];
    for (int k = 0; k < NTERMS; ++k) acc[k] = 0.0;
    for (int i = chunk_begin[ch] + threadIdx.x; i < chunk_end[ch]; i += blockDim.x) {
        const vec_t<T> qi = C.qA[i];
        const vec_t<T> pi = C.pA[i];
        const vec_t<T> f = C.F[i];
        const double e = eps_value(C.eA[i]);
        const bool fin = finite3(qi) && finite3(pi) && isfinite(e);
        acc[0] += ((double)pi.x * pi.x + (double)pi.y * pi.y + (double)pi.z * pi.z) * (0.5 / (double)C.m);
        acc[2] += e;
        acc[3] += pi.x; acc[4] += pi.y; acc[5] += pi.z;
        acc[6] += R.cv / e;
        acc[7] += (double)f.x * f.x + (double)f.y * f.y + (double)f.z * f.z;
        acc[9] += (e <= 0.0) ? 1.0 : 0.0;
        acc[10] += fin ? 0.0 : 1.0;
        if (fin) {
            // the pair sums of the tiled pass, in the step's precision
            const vec_t<T> ul = C.dp[i];
            acc[1] += 0.5 * (double)ul.x;   // each pair is seen twice
            acc[8] += (double)ul.y;
        }
    }
    __shared__ double sh[NTERMS][OBS_THREADS];
    for (int k = 0; k < NTERMS; ++k) sh[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = OBS_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < NTERMS; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < NTERMS) partial[(size_t)ch * NTERMS + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_obs_reps(const double* __restrict__ partial, const int* __restrict__ rep_chunk_begin,
                           int R, double* __restrict__ out) {
    const int r = blockIdx.x;
    if (r >= R || threadIdx.x >= NTERMS) return;
    double s = 0.0;
    for (int ch = rep_chunk_begin[r]; ch < rep_chunk_begin[r + 1]; ++ch) s += partial[(size_t)ch * NTERMS + threadIdx.x];
    out[(size_t)r * NTERMS + threadIdx.x] = s;
}

// cell coordinates of every particle in id order (diagnostic)
template <class T>
__global__ void k_get_cells(Ctx<T> C, int* __restrict__ out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= C.N) return;
    const RepInfo& R = C.reps[C.rep_of_slot[s]];
    const long long g = (long long)R.part_off + id_of(C.qA[s]);
    const int cc = C.cA[s];
    out[3 * g] = cell_x(cc);
    out[3 * g + 1] = cell_y(cc);
    out[3 * g + 2] = cell_z(cc);
}

// ---------------------------------------------------------------------------
// diagnostics
// ---------------------------------------------------------------------------
__global__ void k_debug_philox(int n, const uint4* __restrict__ ctr, const uint2* __restrict__ key,
                               uint4* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = philox4x32_10(ctr[i], philox_keys(key[i]));
}

template <class T>
__global__ void k_debug_gauss(int n, uint2 seed, const double2* tab, const uint32_t* __restrict__ step,
                              const uint32_t* __restrict__ rep, const uint32_t* __restrict__ a,
                              const uint32_t* __restrict__ b, double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T3<T> g = pair_gauss<T>(philox_keys(seed, tab), step[i], rep[i], a[i], b[i]);
    out[3 * i] = g.x; out[3 * i + 1] = g.y; out[3 * i + 2] = g.z;
}

}  // namespace dpde
