// dpde_force.cuh -- the force pass: conservative forces F(q) on set B (Eq.
// newton), the second Verlet half-kick p += dt/2 F when kick != 0, and the
// lists of the fluctuation/dissipation part:
//   LIST_ALL   every neighbour (j, w = 1 - r/r_cut)           -> nbr
//   LIST_CROSS neighbours in another brick                      -> nbr
//              and forward neighbours in the same brick         -> fwd
//   LIST_FWD   forward neighbours (whole-replica SSA)           -> fwd
//   LIST_OBS   (observables) no lists or forces: sums of v and its Laplacian
// A forward neighbour of i lies in the half stencil (segment > 13) or in i's
// own cell after i. Every path visits the neighbour cells in increasing
// segment s = 9 (dz+1) + 3 (dy+1) + (dx+1) and each cell in slot (= id)
// order, so a forward row lists i's pairs in SSA sequence order.
//
// Two kinds of tile:
//   frame tile  tile_edge^3 cells (the tuning's tile edge). It fixes the
//               arithmetic only: separations are differences of positions
//               shifted into a frame centred on the frame tile, or, where
//               the frame tile's halo holds more than hframe particles,
//               differences of cell offsets shifted by the cell distance.
//   work tile   the part of a frame tile one block computes. Its size follows
//               the shared memory the mean density needs and the number of
//               blocks the chip needs (set_tiles), and never changes a bit.
#pragma once

#include <type_traits>

#include "dpde_kernels.cuh"

namespace dpde {

// Sums and list cursors of one particle. The lists share one buffer, entry
// rows nbr [0, cap) then fwd [cap, 2 cap), so an entry's address is its row
// times the row's bytes (which fit 32 bits) beyond the particle's first.
template <class T>
struct PairOut {
    T fx = 0, fy = 0, fz = 0;
    T u = 0;    // sum of v(r) over the neighbours
    uint32_t nn = 0, nf = 0;   // next rows: nbr (from 0), fwd (from cap)
    char* lists = nullptr;     // row 0 of the particle
};

template <class T>
__device__ __forceinline__ PairOut<T> pair_out(const Ctx<T>& C, int i) {
    PairOut<T> o;
    o.lists = reinterpret_cast<char*>(C.nbr + i);
    o.nf = (uint32_t)C.nbr_cap;
    return o;
}

// 1/sqrt(x) of a normal x: rsqrtf without its scaling of denormals
__device__ __forceinline__ float rsqrt_normal(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_normal(double x) { return rsqrt(x); }
template <class T> __device__ __forceinline__ T min_normal();
template <> __device__ __forceinline__ float min_normal() { return 1.17549435e-38f; }
template <> __device__ __forceinline__ double min_normal() { return 2.2250738585072014e-308; }

// One neighbour j (global slot) of i at separation d with |d|^2 = r2 > 0 and
// ir = 1/r, where hit; nothing otherwise. fwd tells whether j is a forward
// neighbour of i, cross whether j's brick differs from i's. sum: add the
// pair's force and potential (a coincident pair has been dealt with). PLAIN:
// the potential is the soft one and the lists have room. Everything is
// predicated, nothing branches.
template <class T, int LM, bool PLAIN>
__device__ __forceinline__ void force_hit(const Ctx<T>& C, bool hit, bool sum, int j, bool fwd, bool cross, T dx, T dy,
                                          T dz, T r2, T ir, PairOut<T>& o) {
    const T w = T(1) - r2 * ir * C.inv_rc;
    T v, fr, lap;
    if (PLAIN) pair_pot_soft(C.pot, r2, ir, v, fr, lap);
    else pair_pot(C.pot, r2, ir, v, fr, lap);
    if (LM == LIST_OBS) {
        if (hit && sum) {
            o.u += v;
            o.fx += lap;
        }
        return;
    }
    if (hit && sum) {
        o.fx += fr * dx; o.fy += fr * dy; o.fz += fr * dz;
        o.u += v;
    }
    if (LM == LIST_NONE) return;
    const bool to_nbr = hit && (LM == LIST_ALL || (LM == LIST_CROSS && cross));
    const bool to_fwd = hit && (LM == LIST_FWD || (LM == LIST_CROSS && !cross)) && fwd;
    // row of the list buffer: nbr rows from 0, fwd rows from cap
    const uint32_t row = to_nbr ? o.nn : o.nf;
    const uint32_t cap = (uint32_t)C.nbr_cap;
    if ((to_nbr || to_fwd) && (PLAIN || row < (to_nbr ? cap : 2 * cap)))
        *reinterpret_cast<ListEnt<T>*>(o.lists + (uint64_t)row * ((uint32_t)C.N * (uint32_t)sizeof(ListEnt<T>))) =
            ListEnt<T>{j, w};
    if (to_nbr) ++o.nn;
    if (to_fwd) ++o.nf;
}

// 1/r of a pair too close for rsqrt_normal; false (and the potential added)
// where the two coincide, which exerts no force
template <class T>
__device__ __forceinline__ bool close_pair(const Ctx<T>& C, T r2, T& ir, PairOut<T>& o) {
    if (r2 > T(0)) {
        ir = trsqrt(r2);
        return true;
    }
    ir = T(0);
    o.u += pair_pot_at_zero(C.pot);
    return false;
}

template <class T, int LM>
__device__ __forceinline__ void force_finish(const Ctx<T>& C, int i, T half_dt, int kick, PairOut<T>& o) {
    if (LM == LIST_OBS) {
        vec_t<T> ul{};
        ul.x = o.u;
        ul.y = o.fx;
        C.dp[i] = ul;
        return;
    }
    const uint32_t cap = (uint32_t)C.nbr_cap;
    o.nf -= cap;
    if (o.nn > cap || o.nf > cap) {
        flag(C.status, ST_CAPACITY);
        o.nn = min(o.nn, cap);
        o.nf = min(o.nf, cap);
    }
    if (LM == LIST_ALL || LM == LIST_CROSS) C.nbr_n[i] = (int)o.nn;
    if (LM == LIST_CROSS || LM == LIST_FWD) C.fwd_n[i] = (int)o.nf;
    vec_t<T> f;
    f.x = o.fx; f.y = o.fy; f.z = o.fz; f.w = T(0);
    C.F[i] = f;
    // each pair is seen from both sides
    C.upot[i] = T(0.5) * o.u;
    if (kick) {
        vec_t<T> pv = C.pB[i];
        pv.x += half_dt * o.fx; pv.y += half_dt * o.fy; pv.z += half_dt * o.fz;
        C.pB[i] = pv;
    }
}

// The frame of a frame tile: its centre cell (unwrapped cell coordinates), or
// rel for cell-relative separations.
struct ForceFrame {
    int cx, cy, cz;
    bool rel;
};

// A particle's coordinate in the frame: its cell offset plus the shift of its
// (unwrapped) cell, c cells from the centre
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float frame_shift(float c, float l) { return __fmul_rn(c, l); }
__device__ __forceinline__ double frame_shift(double c, double l) { return __dmul_rn(c, l); }
template <class T> __device__ __forceinline__ T in_frame(T o, int c, T l) { return add_rn(o, frame_shift((T)c, l)); }

// Per-particle path on global memory (work tiles whose halo does not fit in
// shared memory even in the second launch): the same separations.
template <class T, int LM>
__device__ void force_one_global(const Ctx<T>& C, int i, const ForceFrame& fr, T half_dt, int kick) {
    const RepInfo& R = C.reps[C.rep_of_slot[i]];
    vec_t<T> qi = C.qB[i];
    const int cc = C.cB[i];
    const int cx = cell_x(cc), cy = cell_y(cc), cz = cell_z(cc);
    const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
    const T lx = cell_len<T>(R, 0), ly = cell_len<T>(R, 1), lz = cell_len<T>(R, 2);
    const int* bt = brick_tab(C.tab, R);
    const int bx = __ldg(bt + cx), by = __ldg(bt + nx + cy), bz = __ldg(bt + nx + ny + cz);
    if (!fr.rel) {
        qi.x = in_frame(qi.x, cx - fr.cx, lx);
        qi.y = in_frame(qi.y, cy - fr.cy, ly);
        qi.z = in_frame(qi.z, cz - fr.cz, lz);
    }
    PairOut<T> o = pair_out(C, i);
    for (int sg = 0; sg < 27; ++sg) {
        const int dxc = sg % 3 - 1, dyc = (sg / 3) % 3 - 1, dzc = sg / 9 - 1;
        int x = cx + dxc, y = cy + dyc, z = cz + dzc;
        if (R.walls && (z < 0 || z >= nz)) continue;   // nothing beyond a wall
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
        const bool cross = __ldg(bt + x) != bx || __ldg(bt + nx + y) != by || __ldg(bt + nx + ny + z) != bz;
        const int c = cell_index(C.tab, R, x, y, z);
        const int e = C.start[c + 1];
        for (int j = C.start[c]; j < e; ++j) {
            if (j == i) continue;
            vec_t<T> qj = C.qB[j];
            T ddx, ddy, ddz;
            if (fr.rel) {
                ddx = (qi.x - qj.x) - shift<T>(dxc, lx);
                ddy = (qi.y - qj.y) - shift<T>(dyc, ly);
                ddz = (qi.z - qj.z) - shift<T>(dzc, lz);
            } else {
                ddx = qi.x - in_frame(qj.x, cx + dxc - fr.cx, lx);
                ddy = qi.y - in_frame(qj.y, cy + dyc - fr.cy, ly);
                ddz = qi.z - in_frame(qj.z, cz + dzc - fr.cz, lz);
            }
            const T r2 = ddx * ddx + ddy * ddy + ddz * ddz;
            if (!(r2 < C.rc2)) continue;
            T ir = rsqrt_normal(r2);
            const bool sum = r2 >= min_normal<T>() || close_pair(C, r2, ir, o);
            force_hit<T, LM, false>(C, true, sum, j, sg > 13 || (sg == 13 && j > i), cross, ddx, ddy, ddz, r2, ir, o);
        }
    }
    force_finish<T, LM>(C, i, half_dt, kick, o);
}

// The tiled pass. A block stages its work tile's halo (one cell around) in
// shared memory in x-fastest halo-cell order (slot order inside a cell): the
// exact position hq in the arithmetic's frame with the slot. In this layout j is a
// forward neighbour of i exactly when its halo index is larger, and the
// candidates of a particle are nine contiguous ranges (the three x-cells of
// each (dy, dz) row), walked in (segment, slot) order by a thread per own
// particle.
//
// The pass is bound by instruction issue. Candidates are tested in float,
// four at a time, against a radius a little larger than the cutoff, and
// listed (12.6 of ~94 at density 3, and the particle itself); the listed ones
// are then tested and computed in the exact arithmetic, in list order, so
// sums and lists come out in the order of a plain walk, the warp going
// through its lists together and without branches. At 1M and density 3: 161
// warp instructions a particle on 25 of 32 lanes (the rows of neighbouring
// cells differ in length), 72 % of the issue slots at four blocks an SM.
//
// Measured against one block per frame tile with hits processed row by row:
// 4M at density 3 (Hybrid) 834 -> 644 us, SER lists at 1M 207 -> 176 us,
// 108,000 particles 61 -> 38 us, 1,000 in FP64 484 -> 44 us (one tile took
// them all, on one SM); Lennard-Jones at 18 particles a cell, whose frame
// tiles fit no SM and went particle by particle through global memory,
// 30.5 ms -> 0.22 ms.
constexpr int TILE_EDGE = 6;       // default tile edge (cells); the autotuner picks 4..8
constexpr int TILE_EDGE_MAX = 8;
constexpr int FORCE_HALO_EDGE = TILE_EDGE_MAX + 2;
constexpr int FORCE_WARPS_MAX = 8;
constexpr int FORCE_HITS = 46;        // candidates listed per particle before they are processed
constexpr int FORCE_SPAN = 20;        // candidates tested between two looks at the lists' room
constexpr int FORCE_LSTRIDE = 50;     // 16-bit entries between two threads' lists: 25 words, so that lists lie in distinct banks
constexpr int FORCE_LIST = 32 * FORCE_LSTRIDE;   // entries of a warp's lists

// Shared-memory shape of a launch: halo particles staged (a multiple of 4),
// halo cells and own cells of the largest work tile; wide: float positions
// are staged beside the exact ones. filter2: square of the filter's radius,
// which covers the rounding of the float coordinates (under 1e-6 of a tile),
// far below 1e-4 of the cutoff; NaN, which lets every candidate pass, where
// the square of a cutoff in FP64 lies near the ends of a float's range (a
// product by a unit per staged coordinate cost the FP64 pass 4 %).
struct ForceShape {
    int hcap, nhc, noc, wide;
    float filter2;
};

template <class T>
__host__ __device__ inline size_t force_smem(const ForceShape& S, int warps) {
    return (size_t)S.hcap * (sizeof(vec_t<T>) + (sizeof(T) != 4 || S.wide ? 16 : 0) + 2 + 2) + (size_t)(S.nhc + S.noc) * 8 +
           (size_t)warps * FORCE_LIST * 2 + (size_t)(S.nhc + 1) * 4 + 32;
}

__device__ __forceinline__ int slot_bits(const float4& q) { return __float_as_int(q.w); }
__device__ __forceinline__ int slot_bits(const d4& q) { return (int)__double_as_longlong(q.w); }

// One work tile on the calling block. A work tile whose halo holds more than
// S.hcap particles is appended to `defer` when that list is given (a second
// launch with a larger capacity takes it), else computed through the global
// path.
template <class T, int LM>
__device__ __forceinline__ void force_tile_run(const Ctx<T>& C, int tile, const int4* __restrict__ tile_org,
                                               const int4* __restrict__ tile_dim, T half_dt, int kick,
                                               const ForceShape& S, const FrameTiles& F, int* defer, int* ndefer) {
    // (aligned by declaration, not by arithmetic on the address, which would
    // turn every access into a generic one)
    extern __shared__ __align__(32) unsigned char force_mem[];
    __shared__ int sh[32];
    __shared__ int s_row[TILE_EDGE_MAX * TILE_EDGE_MAX + 1];
    __shared__ T s_shift[3][FORCE_HALO_EDGE];
    using vec = vec_t<T>;
    const int4 org = tile_org[tile];
    const int4 dim = tile_dim[tile];
    const RepInfo& R = C.reps[org.x];
    const int HX = dim.x + 2, HY = dim.y + 2, HZ = dim.z + 2;
    const int HC = HX * HY * HZ;
    const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    vec* hq = reinterpret_cast<vec*>(force_mem);
    // float positions of the filter: hq itself, or a float copy in FP64 or
    // where hq holds cell offsets
    float4* fq = sizeof(T) == 4 && !S.wide ? reinterpret_cast<float4*>(hq) : reinterpret_cast<float4*>(hq + S.hcap);
    int2* cinfo = reinterpret_cast<int2*>(fq + S.hcap);   // halo cell: (first slot - first halo index, code)
    int2* obr = cinfo + S.nhc;
    // lists, a warp's after another's, a thread's own from mylist
    unsigned short* mylist = reinterpret_cast<unsigned short*>(obr + S.noc) + (size_t)tid * FORCE_LSTRIDE;
    int* hstart = reinterpret_cast<int*>(reinterpret_cast<unsigned short*>(obr + S.noc) + (size_t)nwarp * FORCE_LIST);
    unsigned short* cell = reinterpret_cast<unsigned short*>(hstart + S.nhc + 1);   // halo cell of a halo particle
    unsigned short* own = cell + S.hcap;
    // 1. cells of the halo: counts and starts
    const float iHX = 1.0f / (float)HX, iHY = 1.0f / (float)HY;
    for (int h = tid; h < HC; h += blockDim.x) {
        const int row = small_div(h, iHX), hx = h - row * HX, hz = small_div(row, iHY), hy = row - hz * HY;
        int x = org.y + hx - 1, y = org.z + hy - 1, z = org.w + hz - 1;
        const bool use = !(R.walls && (z < 0 || z >= nz));   // beyond a wall: an empty halo cell
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
        int a = 0, n = 0;
        if (use) {
            const int c = cell_index(C.tab, R, x, y, z);
            a = C.start[c];
            n = C.start[c + 1] - a;
        }
        cinfo[h] = make_int2(a, hx | (hy << 4) | (hz << 8));
        hstart[h] = n;
    }
    // slot range of each own cell's brick (LIST_CROSS tells cross pairs by it)
    const int nown = dim.x * dim.y * dim.z;
    if (LM == LIST_CROSS) {
        const int* bt = brick_tab(C.tab, R);
        const int kc = R.k[0] * R.k[1] * R.k[2];
        for (int c = tid; c < nown; c += blockDim.x) {
            const int bx = __ldg(bt + org.y + c % dim.x), by = __ldg(bt + nx + org.z + (c / dim.x) % dim.y),
                      bz = __ldg(bt + nx + ny + org.w + c / (dim.x * dim.y));
            const int c0 = R.cell_off + ((bz * R.B[1] + by) * R.B[0] + bx) * kc;
            const int s0 = C.start[c0];
            obr[c] = make_int2(s0, C.start[c0 + kc] - s0);
        }
    }
    __syncthreads();
    // 2. exclusive scan of the halo counts (a run of cells per thread)
    {
        const int per = (HC + blockDim.x - 1) / blockDim.x;
        const int h0 = min(HC, tid * per), h1 = min(HC, h0 + per);
        int run = 0;
        for (int h = h0; h < h1; ++h) run += hstart[h];
        int total;
        int ex = block_exclusive_scan(run, sh, total);
        for (int h = h0; h < h1; ++h) {
            const int v = hstart[h];
            hstart[h] = ex;
            ex += v;
        }
        if (tid == 0) hstart[HC] = total;
    }
    __syncthreads();
    const int H = hstart[HC];
    const T lx = cell_len<T>(R, 0), ly = cell_len<T>(R, 1), lz = cell_len<T>(R, 2);
    const int4 fo = F.org[dim.w];
    ForceFrame fr;
    fr.rel = LM == LIST_OBS || F.rel[dim.w] != 0;   // the observables' pairs are formed cell by cell throughout
    fr.cx = fo.y - 1 + (min(F.edge, nx - fo.y) + 2) / 2;
    fr.cy = fo.z - 1 + (min(F.edge, ny - fo.z) + 2) / 2;
    fr.cz = fo.w - 1 + (min(F.edge, nz - fo.w) + 2) / 2;
    if (H > S.hcap) {
        if (defer) {
            if (tid == 0) defer[atomicAdd(ndefer, 1)] = tile;
            return;
        }
        // eight threads an own cell (one left most of the block idle)
        for (int u = tid; u < nown << 3; u += blockDim.x) {
            const int c = u >> 3;
            const int h = ((c / (dim.x * dim.y) + 1) * HY + (c / dim.x) % dim.y + 1) * HX + c % dim.x + 1;
            const int g = cinfo[h].x, n = hstart[h + 1] - hstart[h];
            for (int k = u & 7; k < n; k += 8) force_one_global<T, LM>(C, g + k, fr, half_dt, kick);
        }
        return;
    }
    // raw: hq holds cell offsets (a cell-by-cell tile, where there is room
    // for the filter's positions beside them; else they are read again)
    const bool raw = fr.rel && (sizeof(T) != 4 || S.wide);
    // 3. stage the halo particles, a thread per particle: the cell of each
    //    first, then its frame position
    for (int h = tid; h < HC; h += blockDim.x) {
        const int b = hstart[h], e = hstart[h + 1];
        cinfo[h].x -= b;
        for (int k = b; k < e; ++k) cell[k] = (unsigned short)h;
    }
    if (tid < 3 * FORCE_HALO_EDGE) {
        const int d = tid / FORCE_HALO_EDGE, k = tid % FORCE_HALO_EDGE;
        const int c = (d == 0 ? org.y - fr.cx : (d == 1 ? org.z - fr.cy : org.w - fr.cz)) + k - 1;
        s_shift[d][k] = frame_shift((T)c, d == 0 ? lx : (d == 1 ? ly : lz));
    }
    __syncthreads();
    for (int k = tid; k < H; k += blockDim.x) {
        const int2 ci = cinfo[cell[k]];
        const int g = ci.x + k;
        vec q = C.qB[g];
        const T x = add_rn(q.x, s_shift[0][ci.y & 15]), y = add_rn(q.y, s_shift[1][(ci.y >> 4) & 15]),
                z = add_rn(q.z, s_shift[2][ci.y >> 8]);
        if (sizeof(T) != 4 || S.wide) fq[k] = make_float4((float)x, (float)y, (float)z, 0.0f);
        if (!raw) {
            q.x = x; q.y = y; q.z = z;
        }
        set_id(q, (uint32_t)g);
        hq[k] = q;
    }
    // 4. the own particles in halo order: offsets of the own rows (at most
    //    64) by the first warp, then a thread per own cell
    const int nrow = dim.y * dim.z;
    if (tid < 32) {
        int carry = 0;
        for (int r0 = 0; r0 < nrow; r0 += 32) {
            const int r = r0 + tid;
            int n = 0;
            if (r < nrow) {
                const int h = ((r / dim.y + 1) * HY + r % dim.y + 1) * HX;
                n = hstart[h + dim.x + 1] - hstart[h + 1];
            }
            int x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (tid >= o) x += y;
            }
            if (r < nrow) s_row[r] = carry + x - n;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (tid == 0) s_row[nrow] = carry;
    }
    __syncthreads();
    for (int c = tid; c < nown; c += blockDim.x) {
        const int r = c / dim.x, cx = c - r * dim.x;
        const int h = ((r / dim.y + 1) * HY + r % dim.y + 1) * HX + 1;
        const int b = hstart[h + cx], e = hstart[h + cx + 1], at = s_row[r] + b - hstart[h];
        for (int k = b; k < e; ++k) own[at + k - b] = (unsigned short)k;
    }
    __syncthreads();
    const float wide2 = S.filter2;
    const bool fast = !fr.rel && C.pot.kind == 0;
    // 5. a thread per own particle
    const int no = s_row[nrow];
    for (int k0 = warp * 32; k0 < no; k0 += nwarp * 32) {
        const bool act = k0 + lane < no;
        const int hi = own[act ? k0 + lane : k0];
        const uint32_t code = (uint32_t)cinfo[cell[hi]].y;
        const vec qi = hq[hi];
        const int i = slot_bits(qi);
        const int icx = (int)(code & 15), icy = (int)((code >> 4) & 15), icz = (int)(code >> 8);
        int2 br = make_int2(0, 0);
        if (LM == LIST_CROSS) br = obr[((icz - 1) * dim.y + icy - 1) * dim.x + icx - 1];
        const float4 fi = fq[hi];
        auto near = [&](int j) {
            const float4 c = fq[j];
            const float dx = fi.x - c.x, dy = fi.y - c.y, dz = fi.z - c.z;
            return !(dx * dx + dy * dy + dz * dz >= wide2);
        };
        PairOut<T> o = pair_out(C, i);
        // the listed candidates of my particle, n of them, in the exact
        // arithmetic; the warp stays together for np passes
        auto drain = [&](int n, int np, auto plain) {
            constexpr bool PLAIN = decltype(plain)::value;   // in the frame; see force_hit
#pragma unroll 2
            for (int p = 0; p < np; ++p) {
                const int hj = p < n ? (int)mylist[p] : hi;
                const vec qj = hq[hj];
                T ddx = qi.x - qj.x, ddy = qi.y - qj.y, ddz = qi.z - qj.z;
                bool hit = hj != hi;
                if (!PLAIN && fr.rel) {
                    if (!raw) {
                        const vec a = C.qB[i], b = C.qB[slot_bits(qj)];
                        ddx = a.x - b.x; ddy = a.y - b.y; ddz = a.z - b.z;
                    }
                    const int cj = cinfo[cell[hj]].y;
                    const int dx = (cj & 15) - icx, dy = ((cj >> 4) & 15) - icy, dz = (cj >> 8) - icz;
                    ddx -= shift<T>(dx, lx);
                    ddy -= shift<T>(dy, ly);
                    ddz -= shift<T>(dz, lz);
                }
                const T r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                hit = hit && r2 < C.rc2;
                T ir = rsqrt_normal(r2);
                bool sum = true;
                if (hit && !(r2 >= min_normal<T>())) sum = close_pair(C, r2, ir, o);   // rare
                const int j = slot_bits(qj);
                force_hit<T, LM, PLAIN>(C, hit, sum, j, hj > hi, (unsigned)(j - br.x) >= (unsigned)br.y, ddx, ddy, ddz,
                                        r2, ir, o);
            }
        };
        unsigned short* end = mylist;   // end of my list
        for (int row = 0; row < 9; ++row) {
            const int c = ((icz + row / 3 - 1) * HY + icy + row % 3 - 1) * HX + icx - 1;
            int j = act ? hstart[c] : 0;
            const int je = act ? hstart[c + 3] : 0;
            for (;;) {
                // FORCE_SPAN candidates at most, four independent ones at a
                // time; every candidate is written to the next free place
                // and the place kept on a hit (no branch per hit)
                const int stop = min(je, j + FORCE_SPAN);
                for (; j + 4 <= stop; j += 4) {
                    const bool h0 = near(j), h1 = near(j + 1), h2 = near(j + 2), h3 = near(j + 3);
                    *end = (unsigned short)j;
                    end += h0;
                    *end = (unsigned short)(j + 1);
                    end += h1;
                    *end = (unsigned short)(j + 2);
                    end += h2;
                    *end = (unsigned short)(j + 3);
                    end += h3;
                }
                for (; j < stop; ++j) {
                    *end = (unsigned short)j;
                    end += near(j);
                }
                const int n = (int)(end - mylist);
                const bool more = __any_sync(0xffffffffu, j < je);
                const bool full = __any_sync(0xffffffffu, n > FORCE_HITS - FORCE_SPAN);
                if (full || (!more && row == 8)) {
                    const int np = __reduce_max_sync(0xffffffffu, n);
                    const bool room =
                        __all_sync(0xffffffffu, (int)o.nn + n <= C.nbr_cap && (int)o.nf + n <= 2 * C.nbr_cap);
                    if (fast && room) drain(n, np, std::integral_constant<bool, true>{});
                    else drain(n, np, std::integral_constant<bool, false>{});
                    end = mylist;
                }
                if (!more) break;
            }
        }
        if (act) force_finish<T, LM>(C, i, half_dt, kick, o);
    }
}

template <class T, int LM>
__global__ void __launch_bounds__(32 * FORCE_WARPS_MAX, sizeof(T) == 4 ? 4 : 2) k_force_tile(Ctx<T> C, const int4* __restrict__ tile_org,
                                                                     const int4* __restrict__ tile_dim, T half_dt,
                                                                     int kick, ForceShape S, FrameTiles F, int* defer,
                                                                     int* ndefer) {
    force_tile_run<T, LM>(C, blockIdx.x, tile_org, tile_dim, half_dt, kick, S, F, defer, ndefer);
}

// The deferred work tiles (dense regions), persistent blocks with a larger
// halo capacity; a tile beyond even that takes the global path.
template <class T, int LM>
__global__ void __launch_bounds__(32 * FORCE_WARPS_MAX) k_force_tile_dense(Ctx<T> C, const int4* __restrict__ tile_org,
                                                                           const int4* __restrict__ tile_dim,
                                                                           T half_dt, int kick, ForceShape S,
                                                                           FrameTiles F, const int* __restrict__ defer,
                                                                           const int* __restrict__ ndefer) {
    const int n = *ndefer;
    for (int u = blockIdx.x; u < n; u += gridDim.x) {
        force_tile_run<T, LM>(C, defer[u], tile_org, tile_dim, half_dt, kick, S, F, nullptr, nullptr);
        __syncthreads();
    }
}

// The observables' pair sums of very sparse systems, a thread per particle on
// global memory: a tile's cost per halo cell outweighs its particles' there.
// Bound by the scattered reads of the cell starts, so of the three x-cells of
// a row, where they are neighbours in memory, the first start and the last end
// are read, all rows at once, and the few particles found tell their cell
// (54 reads a particle otherwise). Us a call by tiles / by particles: 300,000
// particles at density 0.02 590 / 123, at 0.1 217 / 121, 1.5M at 0.1 818 / 308,
// at 0.5 435 / 370.
template <class T>
__global__ void k_obs_sparse(Ctx<T> C) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C.N) return;
    const RepInfo& R = C.reps[C.rep_of_slot[i]];
    const vec_t<T> qi = C.qB[i];
    const int cc = C.cB[i];
    const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
    const int cx = cell_x(cc);
    const int xm = cx == 0 ? nx - 1 : cx - 1, xp = cx == nx - 1 ? 0 : cx + 1;
    const int c00 = cell_index(C.tab, R, cx, 0, 0);   // (a cell's index is a sum over its coordinates)
    const int om = cell_index(C.tab, R, xm, 0, 0) - c00, op = cell_index(C.tab, R, xp, 0, 0) - c00;
    const bool joined = om == -1 && op == 1;
    int first[9], b[9], e[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        int y = cell_y(cc) + r % 3 - 1, z = cell_z(cc) + r / 3 - 1;
        const bool use = !(R.walls && (z < 0 || z >= nz));   // nothing beyond a wall
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
        first[r] = use ? cell_index(C.tab, R, cx, y, z) : -1;
        b[r] = e[r] = 0;
        if (use && joined) {
            b[r] = C.start[first[r] - 1];
            e[r] = C.start[first[r] + 2];
        }
    }
    const T lx = cell_len<T>(R, 0), ly = cell_len<T>(R, 1), lz = cell_len<T>(R, 2);
    PairOut<T> o = pair_out(C, i);
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const T sy = shift<T>(r % 3 - 1, ly), sz = shift<T>(r / 3 - 1, lz);
        auto visit = [&](int j, int dxc) {
            if (j == i) return;
            const vec_t<T> qj = C.qB[j];
            const T dx = (qi.x - qj.x) - shift<T>(dxc, lx), dy = (qi.y - qj.y) - sy, dz = (qi.z - qj.z) - sz;
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < C.rc2)) return;
            T ir = rsqrt_normal(r2);
            const bool sum = r2 >= min_normal<T>() || close_pair(C, r2, ir, o);
            force_hit<T, LIST_OBS, false>(C, true, sum, j, false, false, dx, dy, dz, r2, ir, o);
        };
        for (int j = b[r]; j < e[r]; ++j) visit(j, cell_x(C.cB[j]) - cx);
        if (!joined && first[r] >= 0)
            for (int d = -1; d <= 1; ++d) {
                const int c = first[r] + (d < 0 ? om : (d > 0 ? op : 0));
                for (int j = C.start[c]; j < C.start[c + 1]; ++j) visit(j, d);
            }
    }
    force_finish<T, LIST_OBS>(C, i, T(0), 0, o);
}

}  // namespace dpde
