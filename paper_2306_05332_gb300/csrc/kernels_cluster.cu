// The coarse end of the V-cycle in one launch (Sec. 2.1 steps 2c-2e and 3, Eq.
// RKL_intermediate_source, App. A.5): a thread-block cluster holds the levels
// B .. C (C the coarsest) in shared memory and runs, without touching global
// memory between them, on every level the pre-smoothing from e = 0, the residual
// and its restriction (mean removed when every axis is periodic, Eq.
// source_modification), on level C the accelerated RKL1 solve (schedule s_k,
// stopped by the coarse tolerance), and on the way back the prolongation and the
// post-smoothing.  Smoothers: RKL super-steps or red-black Gauss-Seidel / SOR
// sweeps.
//
// What bounds it.  These levels are far too small to fill the chip: launched
// level by level, every stage cost a launch (2.5 - 3.1 us in a graph, whatever its
// size), and a level's V-cycle share at the default N_pre = 2, N_post = 1, s = 3 is
// 13 launches.  Here a stage costs a chain of shared-memory loads and FMAs and a
// barrier: 0.67 us on a 32^3 level over 16 CTAs, 0.25 us on 8^3 and below (a whole
// 32^3 solve with the default options: 2.11 ms level by level, 0.79 ms resident).
//
// Cells.  A thread owns two cells of a row in two neighbouring planes (2 x 2 cells of a
// two-dimensional level) through all stages: iterate, right-hand side, Y0, Z0 and
// Y_{j-2} stay in its registers, and a stage reads only the strips around its cells
// from shared memory.  The threads of rows 2J and 2J + 1 are neighbouring lanes, so a
// restriction is their two sums and one shuffle.  (A whole 2 x 2 x 2 block per thread
// took 590 - 610 cycles for a stage of a 4^3 or 8^3 level, the chain of one thread's
// instructions.)
//
// Levels.  A large level is cut along z into slabs of plane pairs over the CTAs of
// the cluster ("split"): a thread on a slab's face also stores its strips into the
// neighbouring CTA's ghost plane through distributed shared memory, counted on a
// barrier there (st.async).  A small level (up to kTailWhole cells;
// FP64, whose arithmetic an SM issues at 1/64 of the FP32 rate, up to kTailWhole64)
// is held whole in every CTA: the same arithmetic on the same data, so every CTA
// takes the same stop decisions (sums in a fixed order), a stage ends with a block
// barrier (the smallest levels run in four warps with a barrier of their own or in
// one warp without any), and each CTA holds every coarse plane that its prolongation
// needs.  On a split level a stage ends when the ghost planes of both neighbours
// have arrived.
//
// Resident solve.  Where level 0 itself is among these levels, a mixed solve's whole
// inner loop runs in the launch: phi and the carried FP64 residual stay in shared
// memory, and after each V-cycle the update phi += e, r -= A_0 e (the arithmetic of
// the update kernel), the norm and the decision to go on are taken here too.
//
// Stages alternate between two buffers, so that a stage reads one and writes the
// other.  Boundaries: a neighbour beyond a Dirichlet wall is the thread's own cell
// with the sign -1 (Eq. error_ghost), beyond a periodic one the cell on the other
// side (Eq. periodic); the sign enters by an FMA, with no branch.
//
// A two-dimensional level (nx, ny) runs as nx x 1 x ny: its second axis is the one
// that is split.
#include "sg_internal.cuh"
#include "sg_update.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

namespace cg = cooperative_groups;

namespace sg {

namespace {

constexpr int kTailMaxNC = 16;           // CTAs per cluster (16: a non-portable size, where the device allows it)
constexpr size_t kSmemLimit = 227u * 1024u - 5120u;   // dynamic shared memory per CTA, next to the static tables
constexpr int kMuTable = 128;            // entries of the table of mu_j of the coarse solve
constexpr int kSchedTable = 64;          // entries of its schedule kept in shared memory

template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

__device__ __forceinline__ float fmat(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmat(double a, double b, double c) { return fma(a, b, c); }

// Pairs of cells, each cell by scalar operations: the packed f32x2 instructions
// need their scalar factors as register pairs, and the moves that build those cost
// more than the arithmetic they save here (106 K warp instructions a CTA of the
// 32^3 .. 2^3 launch with them).
__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }
template <typename T, typename V>
__device__ __forceinline__ V fma2(T a, V b, V c) {
    return mk2(fmat(a, b.x, c.x), fmat(a, b.y, c.y));
}
template <typename T, typename V>
__device__ __forceinline__ V mul2(T a, V b) {
    return mk2(a * b.x, a * b.y);
}
template <typename V>
__device__ __forceinline__ V add2(V a, V b) {
    return mk2(a.x + b.x, a.y + b.y);
}
template <typename V>
__device__ __forceinline__ V neg2(V v) {
    v.x = -v.x;
    v.y = -v.y;
    return v;
}

// Plane pairs of a split level: rank r owns pairs [first(r), first(r + 1)).
__host__ __device__ __forceinline__ int first_pair(int r, int np, int nc) { return r * np / nc; }

// a / n with inv = 1 / n in FP32, for a + 1/2 < 2^22: (a + 1/2) / n is at least 1 / (2 n)
// away from an integer, and inv and the product together are off by less than 2^-23 of it.
// The largest a here is nc plane pairs less one, below 16 x 2^15 for rows of 2^16 cells.
__host__ __device__ __forceinline__ int quick_div(int a, float inv) { return int((float(a) + 0.5f) * inv); }

// The CTA that owns plane pair p.
template <typename T>
__host__ __device__ __forceinline__ int owner_of(const TailLevel<T>& L, int p, int nc) {
    return quick_div((p + 1) * nc - 1, L.inv_pairs);
}

// What a thread needs of the level it works on.  A thread owns the cells
// (2q, 2q + 1) of row j in the planes 2P and 2P + 1 of its slab; on a
// three-dimensional level the threads of rows 2J and 2J + 1 are neighbouring
// lanes, so the two of them hold one 2 x 2 x 2 block.
template <typename T, bool TWOD>
struct Here {
    bool act, split;
    int group;
    int q, j, P, p0;                            // p0: first plane pair of the slab
    int row, plane;
    int o, oym, oyp, ozm, ozp, oxl, oxr;        // offsets in a buffer of the cells and of the strips around them
    int oys, oyn;                               // the y neighbours again: the one with sign sys and the other
    T sym, syp, szm, szp, sxl, sxr, sys;        // -1 across a Dirichlet wall, else 1
    int to_lo, to_hi, lo_off, hi_off;           // CTA (-1: none) and offset of the ghost strips this thread feeds
    unsigned far_lo, far_hi;                    // their addresses in the cluster's shared memory (0: none) ...
    unsigned bar_lo, bar_hi;                    // ... and the barriers that their arrival counts on
    unsigned bytes;                             // ghost bytes that this CTA receives in an exchange
    int fo, fplane;                             // offset in the right-hand side, its plane
    T hx, hy, hz, md;
};

template <typename T, bool TWOD>
__host__ __device__ __forceinline__ Here<T, TWOD> make_here(const TailParams<T>& p, const TailLevel<T>& L, int rank,
                                                            int nc, int tid) {
    Here<T, TWOD> h;
    const int np = L.nz >> 1, nq = L.nx >> 1, ny = TWOD ? 1 : L.ny;
    h.split = L.split != 0;
    h.group = L.group;
    h.p0 = h.split ? L.first[rank] : 0;
    const int pairs = (h.split ? L.first[rank + 1] : np) - h.p0;
    h.act = tid < nq * ny * pairs;
    const int t = h.act ? tid : 0;
    if (TWOD) {
        h.P = quick_div(t, L.inv_nq);
        h.q = t - h.P * nq;
        h.j = 0;
    } else {
        const int u = quick_div(t >> 1, L.inv_nq);          // J of this slab's pairs, one after the other
        h.q = (t >> 1) - u * nq;
        h.P = quick_div(2 * u, L.inv_ny);
        h.j = 2 * u - h.P * ny + (t & 1);
    }
    h.row = L.row;
    h.plane = L.row * ny;
    const int gz = h.split ? 1 : 0;             // ghost planes below the slab
    h.o = (2 * h.P + gz) * h.plane + h.j * h.row + 2 * h.q;
    const bool px = p.per[0] != 0, py = p.per[1] != 0, pz = p.per[2] != 0;
    h.sxl = h.sxr = h.sym = h.syp = h.szm = h.szp = T(1);
    h.oxl = h.o - 1;
    if (h.q == 0) {
        h.oxl = px ? h.o + L.nx - 1 : h.o;
        if (!px) h.sxl = T(-1);
    }
    h.oxr = h.o + 2;
    if (h.q == nq - 1) {
        h.oxr = px ? h.o - (L.nx - 2) : h.o + 1;
        if (!px) h.sxr = T(-1);
    }
    h.oym = h.o - h.row;
    h.oyp = h.o + h.row;
    if (!TWOD) {
        if (h.j == 0) {
            h.oym = py ? h.o + (ny - 1) * h.row : h.o;
            if (!py) h.sym = T(-1);
        }
        if (h.j == ny - 1) {
            h.oyp = py ? h.o - (ny - 1) * h.row : h.o;
            if (!py) h.syp = T(-1);
        }
    }
    const bool above = h.syp < T(0);            // (a row has one wall at most: ny >= 2)
    h.oys = above ? h.oyp : h.oym;
    h.oyn = above ? h.oym : h.oyp;
    h.sys = above ? h.syp : h.sym;
    h.ozm = h.o - h.plane;
    h.ozp = h.o + 2 * h.plane;
    h.to_lo = h.to_hi = -1;
    h.lo_off = h.hi_off = 0;
    const int gp = h.p0 + h.P;                  // global plane pair
    if (gp == 0 && !pz) {
        h.ozm = h.o;
        h.szm = T(-1);
    } else if (h.split) {
        if (h.P == 0) {                         // feeds the ghost plane above the slab below
            h.to_lo = owner_of(L, gp > 0 ? gp - 1 : np - 1, nc);
            const int there = L.first[h.to_lo + 1] - L.first[h.to_lo];
            h.lo_off = (2 * there + 1) * h.plane + h.j * h.row + 2 * h.q;
        }
    } else if (gp == 0) {
        h.ozm = h.o + (L.nz - 1) * h.plane;
    }
    if (gp == np - 1 && !pz) {
        h.ozp = h.o + h.plane;
        h.szp = T(-1);
    } else if (h.split) {
        if (h.P == pairs - 1) {
            h.to_hi = owner_of(L, gp < np - 1 ? gp + 1 : 0, nc);
            h.hi_off = h.j * h.row + 2 * h.q;
        }
    } else if (gp == np - 1) {
        h.ozp = h.o - (L.nz - 2) * h.plane;
    }
    h.bytes = 0;
    if (h.split && pairs > 0)
        h.bytes = unsigned((h.p0 > 0 || pz) + (h.p0 + pairs < np || pz)) * unsigned(L.nx * ny) * unsigned(sizeof(T));
    h.fplane = L.nx * ny;
    h.fo = 2 * h.P * h.fplane + h.j * L.nx + 2 * h.q;
    h.hx = L.hx;
    h.hy = L.hy;
    h.hz = L.hz;
    h.md = L.md;
    return h;
}

constexpr int kFourWarps = 128;

// Shared memory of another CTA of the cluster by its 32-bit address.
__device__ __forceinline__ unsigned far_address(const void* p, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
// A store into it whose bytes are counted on the receiver's barrier when they land.
__device__ __forceinline__ void st_far(unsigned a, float2 v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a),
                 "f"(v.x), "f"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_far(unsigned a, double2 v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(a),
                 "d"(v.x), "d"(v.y), "r"(bar)
                 : "memory");
}
// Bounded wait for a phase of a barrier of this CTA (a wait that gives up is
// reported: see the end of the kernel).
constexpr int kTailWaitTries = 1 << 20;
__device__ __forceinline__ bool wait_phase(unsigned bar, unsigned parity) {
    for (int i = 0; i < kTailWaitTries; ++i) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// Launches with a wait that gave up since the library was loaded.
__device__ unsigned int g_tail_wait_timeouts = 0;

template <typename T, bool TWOD>
__global__ void __launch_bounds__(tail_threads<T>()) k_tail_levels(const __grid_constant__ TailParams<T> p) {
    using V = typename Pair<T>::type;
    using H = Here<T, TWOD>;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T* const sm = reinterpret_cast<T*>(sm_raw);
    __shared__ T red[32];
    __shared__ T redc[2][kTailMaxNC];
    __shared__ T mu_tab[kMuTable];
    __shared__ int sched[kSchedTable];
    __shared__ int joined;                       // what the warps left out of the smallest levels missed
    // Level descriptions and stage coefficients in shared memory: indexed reads of
    // the parameter bank in every stage and at every change of level cost more than
    // the arithmetic between them (a stage of a 4^3 level, 16 threads: 795 cycles)
    __shared__ TailLevel<T> lvs[kTailMaxLevels];
    __shared__ T coef[kTailMaxS + 1][4];         // mu, nu, c0 of stage j; the first: 1, 0, 0
    __shared__ LoopState state;
    __shared__ double inv_nn, inv_rden;
    // ghost planes arrive on these, exchange n on barrier n & 1 (a neighbour is at most
    // one exchange ahead: its next one needs this CTA's data of the one before)
    __shared__ unsigned long long xbar[2];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), nc = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31;
    int rslot = 0;
    unsigned xn = 0;                             // exchanges so far, the same count in every CTA
    // After a wait that gave up the thread neither arms a barrier (a phase that is not
    // complete must not be armed again) nor sends; its neighbours give up in their turn.
    bool waits_ok = true;
    __shared__ int gave_up;                      // on CTA 0: some thread of the cluster did
    if (tid == 0) {
        gave_up = 0;
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(&xbar[b]))
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }

    for (int j = tid; j < kMuTable; j += blockDim.x) mu_tab[j] = j > 0 ? T(2) - T(1) / T(j) : T(0);
    for (int j = tid; j < kSchedTable && j < p.max_ss; j += blockDim.x) sched[j] = p.sched[j];
    for (int j = tid; j < int(sizeof(lvs) / sizeof(int)); j += blockDim.x)
        reinterpret_cast<int*>(lvs)[j] = reinterpret_cast<const int*>(p.lv)[j];
    for (int j = 1 + tid; j <= p.s; j += blockDim.x) {
        coef[j][0] = j == 1 ? T(1) : p.mu[j];
        coef[j][1] = j == 1 ? T(0) : p.nu[j];
        coef[j][2] = j == 1 || p.order == 1 ? T(0) : p.c0[j];
    }
    // mu~ tau and gamma~ tau of every level but the coarsest, the product in 64 bits
    for (int n = tid; n < (p.nl - 1) * p.s; n += blockDim.x) {
        const int l = n / p.s, j = n - l * p.s + 1;
        const double tau = p.lv[l].tau;
        reinterpret_cast<V*>(sm + p.lv[l].scaled)[j - 1] =
            mk2(T(p.mut[j] * tau), j == 1 || p.order == 1 ? T(0) : T(p.gt[j] * tau));
    }
    cl.sync();                                   // every CTA runs before a peer writes into it

    auto here = [&](const TailLevel<T>& L) {
        H h = make_here<T, TWOD>(p, L, rank, nc, tid);
        h.far_lo = h.to_lo >= 0 ? far_address(sm + h.lo_off, h.to_lo) : 0u;
        h.far_hi = h.to_hi >= 0 ? far_address(sm + h.hi_off, h.to_hi) : 0u;
        h.bar_lo = h.to_lo >= 0 ? far_address(xbar, h.to_lo) : 0u;
        h.bar_hi = h.to_hi >= 0 ? far_address(xbar, h.to_hi) : 0u;
        return h;
    };
    auto group_threads = [&](int group) -> int {
        return group == 0 ? (int)blockDim.x : min((int)blockDim.x, group == 1 ? kFourWarps : 32);
    };
    auto group_sync = [&](int group) {           // barrier `group` of the CTA
        asm volatile("bar.sync %0, %1;" ::"r"(group), "r"(group_threads(group)) : "memory");
    };
    auto sync = [&](const H& h) {
        if (h.split) cl.sync();
        else group_sync(h.group);
    };
    auto ld = [](const T* a) { return *reinterpret_cast<const V*>(a); };
    auto st = [](T* a, V v) { *reinterpret_cast<V*>(a) = v; };

    // L c - f of the thread's cells c from buffer y, nf = -f, by the second differences of
    // each axis: (lower - 2 c) + upper, in FP64, whose operations count, -2 c + (lower +
    // upper), one fewer.  (Neighbours summed against one term -2 (h_x + h_y + h_z) c take
    // another one or two less, but the rounding of that coefficient acts on c itself and not
    // on its differences: one V-cycle of a smooth 48 x 64 x 56 field was off by
    // 5.0 - 7.1e-7 with it, by 1.2 - 2.1e-7 level by level.)
    auto lap = [&](const H& h, const T* y, const V (&c)[2], const V (&nf)[2], V (&out)[2]) {
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int at = a * h.plane;
            const T xl = y[h.oxl + at], xr = y[h.oxr + at];
            V dx, dz, dy;
            if constexpr (sizeof(T) == 8) {
                dx = fma2(T(-2), c[a], mk2(fmat(h.sxl, xl, c[a].y), fmat(h.sxr, xr, c[a].x)));
                dz = fma2(T(-2), c[a], a == 0 ? fma2(h.szm, ld(y + h.ozm), c[1]) : fma2(h.szp, ld(y + h.ozp), c[0]));
                if constexpr (!TWOD) dy = fma2(T(-2), c[a], fma2(h.sys, ld(y + h.oys + at), ld(y + h.oyn + at)));
            } else {
                const V m2 = mul2(T(-2), c[a]);
                dx = mk2(fmat(h.sxl, xl, m2.x) + c[a].y, fmat(h.sxr, xr, m2.y) + c[a].x);
                dz = add2(a == 0 ? fma2(h.szm, ld(y + h.ozm), m2) : fma2(h.szp, ld(y + h.ozp), m2), c[1 - a]);
                if constexpr (!TWOD) dy = fma2(h.syp, ld(y + h.oyp + at), fma2(h.sym, ld(y + h.oym + at), m2));
            }
            V v = fma2(h.hz, dz, nf[a]);
            if constexpr (!TWOD) v = fma2(h.hy, dy, v);
            out[a] = fma2(h.hx, dx, v);
        }
    };
    // The cells into buffer `off` of this CTA and, on a split level, the slab's faces
    // into the ghost planes of the neighbouring slabs; then the barrier that ends a
    // stage: the group's own, and on a split level the arrival of the ghost planes of
    // exchange xn.  Only neighbours wait for each other (a release / acquire barrier of
    // the whole cluster instead took 700 - 1200 cycles at 128 - 512 threads against
    // 400 - 820).  A thread reads just the ghost strips beside its own cells, before it
    // sends those cells, so data of a neighbour's next exchange cannot overtake a read.
    auto publish = [&](const H& h, auto split, int off, const V (&c)[2]) {
        if constexpr (decltype(split)::value) {
            if (tid == 0 && waits_ok)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(&xbar[xn & 1])),
                             "r"(h.bytes)
                             : "memory");
        }
        if (h.act) {
            T* y = sm + off + h.o;
            st(y, c[0]);
            st(y + h.plane, c[1]);
            if constexpr (decltype(split)::value) {
                if (h.far_lo && waits_ok) st_far(h.far_lo + off * (int)sizeof(T), c[0], h.bar_lo + 8 * (xn & 1));
                if (h.far_hi && waits_ok) st_far(h.far_hi + off * (int)sizeof(T), c[1], h.bar_hi + 8 * (xn & 1));
            }
        }
        group_sync(h.group);
        if constexpr (decltype(split)::value) {
            if (waits_ok)
                waits_ok = wait_phase((unsigned)__cvta_generic_to_shared(&xbar[xn & 1]), (xn >> 1) & 1u);
            ++xn;
        }
    };
    auto publish_any = [&](const H& h, int off, const V (&c)[2]) {
        if (h.split) publish(h, std::true_type{}, off, c);
        else publish(h, std::false_type{}, off, c);
    };
    // sum of v over the level's threads in a fixed order, the same in every CTA
    auto level_sum = [&](const H& h, T v) -> T {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (h.group == 2) return v;
        const int nw = group_threads(h.group) >> 5;
        group_sync(h.group);                     // red is free (previous readers done)
        if (lane == 0) red[tid >> 5] = v;
        group_sync(h.group);
        T t = T(0);
        for (int k = 0; k < nw; ++k) t += red[k];
        if (!h.split) return t;
        rslot ^= 1;                              // a CTA is at most one cluster barrier ahead of a reader
        if (tid < nc) cl.map_shared_rank(&redc[rslot][0], tid)[rank] = t;
        cl.sync();
        t = T(0);
        for (int k = 0; k < nc; ++k) t += redc[rslot][k];
        return t;
    };

    // `count` smoothing steps of level l on the cells c with the iterate published
    // in buffer cur (zero: c = 0, nothing published yet); the result is published.
    // The stages are one loop without branches but its own: every thread of the
    // group computes (those without cells on cell 0's strips), the stores are
    // predicated, the first stage is the general one with mu = 1 and the other
    // factors 0.
    auto smooth_on = [&](auto split, const H& h, const TailLevel<T>& L, int count, bool zero, V (&c)[2],
                         const V (&nf)[2], int& cur) {
        int off = L.buf + cur * L.fld;
        const int flip = (2 * L.buf + L.fld);    // off + other = flip
        if (p.gsrb) {
            // diagonal of each cell's row: -1/h^2 more for each Dirichlet wall it
            // touches (its ghost holds minus the cell)
            const T om = L.omega;
            V inv[2];
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                T d = h.md;
                if ((a == 0 ? h.szm : h.szp) < T(0)) d -= h.hz;
                if (!TWOD && h.sym < T(0)) d -= h.hy;
                if (!TWOD && h.syp < T(0)) d -= h.hy;
                inv[a] = mk2(T(1) / (h.sxl < T(0) ? d - h.hx : d), T(1) / (h.sxr < T(0) ? d - h.hx : d));
            }
#pragma unroll 1
            for (int n = 0; n < 2 * count; ++n) {
                V l[2];
                if (zero && n == 0) {
                    l[0] = nf[0];
                    l[1] = nf[1];
                } else {
                    lap(h, sm + off, c, nf, l);
                }
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    // 2q and 2P are even: cell x of plane a has the parity of x + j + a
                    const bool left = ((a + h.j + n) & 1) == 0;
                    const T x = c[a].x - om * l[a].x * inv[a].x, y = c[a].y - om * l[a].y * inv[a].y;
                    c[a] = mk2(left ? x : c[a].x, left ? c[a].y : y);
                }
                off = flip - off;
                publish(h, split, off, c);
            }
            cur = off == L.buf ? 0 : 1;
            return;
        }
        const V* const scaled = reinterpret_cast<const V*>(sm + L.scaled) - 1;
        V y0[2], z[2], m2[2];
        y0[0] = y0[1] = z[0] = z[1] = m2[0] = m2[1] = mk2(T(0), T(0));
        int js = 1;
#pragma unroll 1
        for (int n = p.s * count; n > 0; --n) {
            const T mu = coef[js][0], nu = coef[js][1], c0 = coef[js][2];
            const V mt_gt = scaled[js];
            V l[2];
            if (zero) {
                l[0] = nf[0];
                l[1] = nf[1];
                zero = false;
            } else {
                lap(h, sm + off, c, nf, l);
            }
            const bool first = js == 1;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                if (first) {
                    y0[a] = c[a];
                    z[a] = l[a];
                }
                // from the small terms to the large ones
                const V v = fma2(mu, c[a], fma2(nu, m2[a], fma2(c0, y0[a], fma2(mt_gt.x, l[a], mul2(mt_gt.y, z[a])))));
                m2[a] = c[a];
                c[a] = v;
            }
            js = js == p.s ? 1 : js + 1;
            off = flip - off;
            publish(h, split, off, c);
        }
        cur = off == L.buf ? 0 : 1;
    };
    auto smooth = [&](const H& h, const TailLevel<T>& L, int count, bool zero, V (&c)[2], const V (&nf)[2], int& cur) {
        if (count == 0 && zero) {
            publish_any(h, L.buf + cur * L.fld, c);
        } else if (h.split) {
            smooth_on(std::true_type{}, h, L, count, zero, c, nf, cur);
        } else {
            smooth_on(std::false_type{}, h, L, count, zero, c, nf, cur);
        }
    };
    auto load_nf = [&](const H& h, const TailLevel<T>& L, V (&nf)[2]) {         // -f of the cells
#pragma unroll
        for (int a = 0; a < 2; ++a) nf[a] = neg2(ld(sm + L.f + h.fo + a * h.fplane));
    };
    auto level_mean = [&](const H& h, const TailLevel<T>& L, V (&nf)[2]) {      // Eq. source_modification
        const T s = h.act ? (nf[0].x + nf[0].y) + (nf[1].x + nf[1].y) : T(0);
        const T mean = level_sum(h, s) * L.inv_cells;
        if (h.act)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                nf[a] = mk2(nf[a].x - mean, nf[a].y - mean);
                st(sm + L.f + h.fo + a * h.fplane, neg2(nf[a]));
            }
    };

    const int nl = p.nl;
    unsigned curs = 0u;                          // bit l: the buffer that holds level l's iterate
    int done = 0;                                // coarse super-steps

    // One V-cycle from e = 0 on the right-hand side of level 0 in shared memory; the
    // thread's cells of e in c
    auto cycle = [&](V (&c)[2]) {
    // ---- down: pre-smoothing from zero, residual, restriction
#pragma unroll 1
    for (int l = 0; l < nl - 1; ++l) {
        const TailLevel<T>& L = lvs[l];
        if (tid >= group_threads(L.group)) break;       // the levels from here on run in fewer warps
        const H h = here(L);
        V nf[2];
        nf[0] = nf[1] = c[0] = c[1] = mk2(T(0), T(0));
        if (h.act) load_nf(h, L, nf);
        if (l > 0 && p.remove_mean) level_mean(h, L, nf);
        int cur = 0;
        smooth(h, L, L.n_pre, true, c, nf, cur);
        curs = (curs & ~(1u << l)) | (unsigned(cur) << l);
        // r = f - L c; its mean over a 2 x 2 x 2 block (2 x 2) is one cell of level l + 1
        const TailLevel<T>& Lc = lvs[l + 1];
        T s = T(0);
        if (h.act) {
            V d[2];
            lap(h, sm + L.buf + cur * L.fld, c, nf, d);
            s = (d[0].x + d[0].y) + (d[1].x + d[1].y);
        }
        if (!TWOD) s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (h.act && (TWOD || !(h.j & 1))) {
            s *= T(-1) / T(TWOD ? 4 : 8);
            const int gp = h.p0 + h.P;           // plane of level l + 1
            const int cy = TWOD ? 1 : Lc.ny;
            if (!Lc.split) {
                const int at = Lc.f + (gp * cy + (h.j >> 1)) * Lc.nx + h.q;
                if (!h.split) sm[at] = s;
                else
                    for (int k = 0; k < nc; ++k) cl.map_shared_rank(sm, k)[at] = s;
            } else {
                const int own = owner_of(Lc, gp >> 1, nc);
                cl.map_shared_rank(sm, own)[Lc.f + ((gp - 2 * Lc.first[own]) * cy + (h.j >> 1)) * Lc.nx + h.q] = s;
            }
        }
        sync(h);
    }

    // ---- level C: accelerated RKL1 from e = 0 (App. A.5)
    {
        const TailLevel<T>& L = lvs[nl - 1];
        if (tid < group_threads(L.group)) {
            const H h = here(L);
            V nf[2], prev[2];
            nf[0] = nf[1] = c[0] = c[1] = prev[0] = prev[1] = mk2(T(0), T(0));
            if (h.act) load_nf(h, L, nf);
            if (nl > 1 && p.remove_mean) level_mean(h, L, nf);
            const T tu = p.tau_unit;
            auto sq = [&](const V (&l)[2]) {
                return fmat(l[0].x, l[0].x, fmat(l[0].y, l[0].y, fmat(l[1].x, l[1].x, l[1].y * l[1].y)));
            };
            T rsq = T(0);
            if (p.tol > T(0)) rsq = level_sum(h, h.act ? sq(nf) : T(0));       // e = 0: the residual is f
            const T tolsq = p.tol * p.tol * rsq;
            int cur = 0;
            done = 0;
            auto solve_on = [&](auto split) {
#pragma unroll 1
                for (int ss = 0; ss < p.max_ss; ++ss) {
                    V l[2];
                    if (p.tol > T(0)) {
                        if (ss > 0) {
                            lap(h, sm + L.buf + cur * L.fld, c, nf, l);
                            rsq = level_sum(h, h.act ? sq(l) : T(0));
                        }
                        if (rsq <= tolsq) break;
                    }
                    const int s = ss < kSchedTable ? sched[ss] : p.sched[ss];
#pragma unroll 1
                    for (int js = 1; js <= s; ++js) {
                        if (js > 1 || (ss > 0 && !(p.tol > T(0)))) {
                            lap(h, sm + L.buf + cur * L.fld, c, nf, l);
                        } else if (ss == 0) {
                            l[0] = nf[0];
                            l[1] = nf[1];
                        }                        // else the residual of the stopping test
                        // Y1 = Y0 + tau_unit (L Y0 - f)
                        // Y_j = mu Y_{j-1} + nu Y_{j-2} + mu tau_unit (L Y_{j-1} - f), mu_1 = 1, nu_1 = 0
                        const T mu = js < kMuTable ? mu_tab[js] : T(2) - T(1) / T(js);
                        const T nu = T(1) - mu, mt = mu * tu;
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            const V v = fma2(mu, c[a], fma2(nu, prev[a], mul2(mt, l[a])));
                            prev[a] = c[a];
                            c[a] = v;
                        }
                        cur ^= 1;
                        publish(h, split, L.buf + cur * L.fld, c);
                    }
                    ++done;
                }
            };
            if (h.split) solve_on(std::true_type{});
            else solve_on(std::false_type{});
            if (done == 0) publish_any(h, L.buf + cur * L.fld, c);     // f = 0 (or no super-step asked for): e = 0
            curs = (curs & ~(1u << (nl - 1))) | (unsigned(cur) << (nl - 1));
        }
    }

    // ---- up: prolongation, correction, post-smoothing
#pragma unroll 1
    for (int l = nl - 2; l >= 0; --l) {
        const TailLevel<T>& L = lvs[l];
        const TailLevel<T>& Lc = lvs[l + 1];
        if (tid >= group_threads(L.group)) continue;
        if (Lc.group > L.group) {                // warps join again and learn what they missed
            if (tid == 0) joined = int(curs >> (l + 1)) & 1;
            group_sync(L.group);
            curs = (curs & ~(1u << (l + 1))) | (unsigned(joined) << (l + 1));
        }
        if (Lc.split) cl.sync();                 // the prolongation reads planes of other CTAs
        const H h = here(L);
        int cur = int((curs >> l) & 1u);
        V nf[2];
        nf[0] = nf[1] = c[0] = c[1] = mk2(T(0), T(0));
        if (h.act) {
            load_nf(h, L, nf);
            const T* y = sm + L.buf + cur * L.fld;
            const int cbuf = Lc.buf + int((curs >> (l + 1)) & 1u) * Lc.fld;
            const int gp = h.p0 + h.P, cnx = Lc.nx, cny = TWOD ? 1 : Lc.ny, cnz = Lc.nz;
            const int crow = Lc.row, cplane = Lc.row * cny;
            // this parent and its neighbours (beyond a wall: minus the parent)
            const bool px = p.per[0] != 0, py = p.per[1] != 0, pz = p.per[2] != 0;
            const int xm = h.q > 0 ? h.q - 1 : (px ? cnx - 1 : 0), xp = h.q < cnx - 1 ? h.q + 1 : (px ? 0 : cnx - 1);
            const T wxm = (h.q == 0 && !px) ? T(-1) : T(1), wxp = (h.q == cnx - 1 && !px) ? T(-1) : T(1);
            const int J = h.j >> 1;
            int Jn = (h.j & 1) ? J + 1 : J - 1;
            T wy = T(1);
            if (Jn < 0) {
                if (!py) wy = T(-1);
                Jn = py ? cny - 1 : 0;
            } else if (Jn >= cny) {
                if (!py) wy = T(-1);
                Jn = py ? 0 : cny - 1;
            }
            V acc[3];                            // x and y interpolated, per coarse plane
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                int K = gp + d - 1;
                T wz = T(1);
                if (K < 0) {
                    if (!pz) wz = T(-1);
                    K = pz ? cnz - 1 : 0;
                } else if (K >= cnz) {
                    if (!pz) wz = T(-1);
                    K = pz ? 0 : cnz - 1;
                }
                const T* e = sm + cbuf;
                if (Lc.split) {
                    const int own = owner_of(Lc, K >> 1, nc);
                    e = cl.map_shared_rank(sm, own) + cbuf + (K - 2 * Lc.first[own] + 1) * cplane;
                } else {
                    e += K * cplane;
                }
                auto xrow = [&](const T* er, T w) {
                    const T v0 = T(3) * er[h.q];
                    return mul2(w, mk2(fmat(wxm, er[xm], v0), fmat(wxp, er[xp], v0)));
                };
                if constexpr (TWOD) acc[d] = xrow(e, wz);
                else acc[d] = fma2(T(3), xrow(e + J * crow, wz), xrow(e + Jn * crow, wz * wy));
            }
            const T w = T(1) / T(TWOD ? 16 : 64);
#pragma unroll
            for (int a = 0; a < 2; ++a)
                c[a] = fma2(w, fma2(T(3), acc[1], acc[2 * a]), ld(y + h.o + a * h.plane));
        }
        cur ^= 1;
        publish_any(h, L.buf + cur * L.fld, c);
        smooth(h, L, L.n_post, false, c, nf, cur);
        curs = (curs & ~(1u << l)) | (unsigned(cur) << l);
    }
    };

    // ---- the right-hand side of the first level; a resident solve's phi and r
    const TailLevel<T>& L0 = lvs[0];
    constexpr bool kMayStay = std::is_same<T, float>::value;
    __shared__ double part[2][kTailMaxNC][2];
    __shared__ float wsq[32], wmx[32];
    __shared__ int go_on;
    auto slab_at = [&](const H& h) { return (size_t)(2 * h.p0) * h.fplane + h.fo; };  // the thread's cells in global memory
    // phi and r of the thread's cells: plane a, phi (0) or r (1)
    auto keep = [&](int a, int which) -> double2& {
        return reinterpret_cast<double2*>(sm + p.resident_off)[(2 * a + which) * (int)blockDim.x + tid];
    };
    const bool stay = kMayStay && p.loop != nullptr;
    {
        const H h = here(L0);
        const size_t at = slab_at(h);
        if (h.act)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                st(sm + L0.f + h.fo + a * h.fplane, ld(p.rhs + at + a * h.fplane));
                if (stay) {
                    keep(a, 0) = *reinterpret_cast<const double2*>(p.phi + at + a * h.fplane);
                    keep(a, 1) = *reinterpret_cast<const double2*>(p.r64 + at + a * h.fplane);
                }
            }
        if (stay && tid == 0) {
            state = *p.loop;
            inv_nn = 1.0 / state.nn;
            inv_rden = 1.0 / state.rden;
        }
    }
    __syncthreads();
    bool go = !stay || state.status == kLoopRunning;
    int slot = 0;
    V c[2];
    // A resident solve repeats the V-cycle, phi += e, r -= A_0 e, its norm and the
    // decision to go on until the recurrence meets the tolerance (every CTA decides
    // from the same sums); otherwise there is one V-cycle.
#pragma unroll 1
    while (go) {
        cycle(c);
        if (!stay) break;
        if constexpr (kMayStay) {
            const H h = here(L0);
            float sq = 0.0f, mx = 0.0f;
            if (h.act) {
                const float* y = sm + L0.buf + int(curs & 1u) * L0.fld;
                const bool uniform = !TWOD && p.ihx2 == p.ihy2 && p.ihy2 == p.ihz2;
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int at = a * h.plane;
                    const float xl = h.sxl * y[h.oxl + at], xr = h.sxr * y[h.oxr + at];
                    const float2 zm = a == 0 ? mul2(h.szm, ld(y + h.ozm)) : c[0];
                    const float2 zp = a == 0 ? c[1] : mul2(h.szp, ld(y + h.ozp));
                    float2 ym = c[a], yp = c[a];
                    if (!TWOD) {
                        ym = mul2(h.sym, ld(y + h.oym + at));
                        yp = mul2(h.syp, ld(y + h.oyp + at));
                    }
                    double2 r = keep(a, 1);
                    if (TWOD) {                  // the second axis of the launch is the level's y axis
                        r.x = update_r<false>(p.ihx2, p.ihy2, p.ihz2, c[a].x, xl, c[a].y, zm.x, zp.x, ym.x, yp.x, r.x);
                        r.y = update_r<false>(p.ihx2, p.ihy2, p.ihz2, c[a].y, c[a].x, xr, zm.y, zp.y, ym.y, yp.y, r.y);
                    } else if (uniform) {
                        r.x = update_r<true>(p.ihx2, p.ihy2, p.ihz2, c[a].x, xl, c[a].y, ym.x, yp.x, zm.x, zp.x, r.x);
                        r.y = update_r<true>(p.ihx2, p.ihy2, p.ihz2, c[a].y, c[a].x, xr, ym.y, yp.y, zm.y, zp.y, r.y);
                    } else {
                        r.x = update_r<false>(p.ihx2, p.ihy2, p.ihz2, c[a].x, xl, c[a].y, ym.x, yp.x, zm.x, zp.x, r.x);
                        r.y = update_r<false>(p.ihx2, p.ihy2, p.ihz2, c[a].y, c[a].x, xr, ym.y, yp.y, zm.y, zp.y, r.y);
                    }
                    keep(a, 1) = r;
                    double2& f = keep(a, 0);
                    f.x += f2d_bits(c[a].x);
                    f.y += f2d_bits(c[a].y);
                    const float2 rf = make_float2(d2f_bits(r.x), d2f_bits(r.y));
                    st(sm + L0.f + h.fo + a * h.fplane, rf);
                    sq = fmaf(rf.x, rf.x, fmaf(rf.y, rf.y, sq));
                    mx = fmaxf(mx, fmaxf(fabsf(rf.x), fabsf(rf.y)));
                }
            }
            // norms: a warp's in FP32, then FP64 in a fixed order
            for (int o = 16; o > 0; o >>= 1) {
                sq += __shfl_xor_sync(0xffffffffu, sq, o);
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
            if (lane == 0) {
                wsq[tid >> 5] = sq;
                wmx[tid >> 5] = mx;
            }
            __syncthreads();
            slot ^= 1;
            if (tid < 32) {
                const int nw = (int)blockDim.x >> 5;
                double a = lane < nw ? double(wsq[lane]) : 0.0;
                float b = lane < nw ? wmx[lane] : 0.0f;
                for (int o = 16; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
                }
                if (lane < nc) {
                    double* there = cl.map_shared_rank(&part[slot][0][0], lane) + 2 * rank;
                    there[0] = a;
                    there[1] = double(b);
                }
            }
            cl.sync();
            if (tid == 0) {
                double a = part[slot][0][0], b = part[slot][0][1];
                for (int k = 1; k < nc; ++k) {
                    a += part[slot][k][0];
                    b = fmax(b, part[slot][k][1]);
                }
                const int m = state.m;
                int cs = 0;
                for (int k = 0; k < done; ++k) cs += k < kSchedTable ? sched[k] : p.sched[k];
                state.coarse_stage_cells += cs * state.coarse_cells;
                bool record;
                go_on = loop_decide(state, sqrt(a * inv_nn) * inv_rden, b, &record) ? 1 : 0;
                if (rank == 0) {
                    if (m < kLoopHistory) p.loop->coarse_ss[m] = done;
                    if (record && m + 1 < kLoopHistory) p.loop->history[m + 1] = state.rel;
                }
            }
            __syncthreads();
            go = go_on != 0;
        }
    }
    {
        const H h = here(L0);
        const size_t at = slab_at(h);
        if (h.act && (h.split || rank == 0))
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                if (stay) *reinterpret_cast<double2*>(p.phi + at + a * h.fplane) = keep(a, 0);
                else st(p.u_out + at + a * h.fplane, c[a]);
            }
        if (rank == 0 && tid == 0) {
            if (stay) *static_cast<LoopState*>(p.loop) = state;
            else if (p.ss_done) *p.ss_done = done;
        }
    }
    if (!waits_ok) {                             // copies on their way land (microseconds) before a CTA ends
        *cl.map_shared_rank(&gave_up, 0) = 1;
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    cl.sync();                                   // peers may still read or write this CTA's memory until here
    // a bounded wait gave up: the solve reports a non-finite residual (from the update's
    // norm; a resident solve from the residual of phi that loop_confirm reads)
    if (rank == 0 && tid == 0 && gave_up) {
        atomicAdd(&g_tail_wait_timeouts, 1u);
        if (stay) p.phi[0] = __longlong_as_double(0x7ff8000000000000ll);
        else p.u_out[0] = T(__int_as_float(0x7fc00000));
    }
}

// Cluster sizes the device schedules with the whole shared memory (bit n: n CTAs),
// per kernel.
template <typename T, bool TWOD>
struct TailCaps {
    static unsigned sizes;
};
template <typename T, bool TWOD>
unsigned TailCaps<T, TWOD>::sizes = 0;

cudaLaunchConfig_t tail_config(int nc, int threads, size_t bytes, cudaStream_t st, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = nc;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <typename T, bool TWOD>
cudaError_t configure_one() {
    auto kern = k_tail_levels<T, TWOD>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e != cudaSuccess) return e;
    // clusters of 16 CTAs are opt-in; where the device refuses, the query below
    // finds none of that size
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        cudaGetLastError();
    unsigned sizes = 2u;
    for (int nc = 2; nc <= kTailMaxNC; ++nc) {
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = tail_config(nc, tail_threads<T>(), kSmemLimit, nullptr, at);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) sizes |= 1u << nc;
        else cudaGetLastError();
    }
    TailCaps<T, TWOD>::sizes = sizes;
    return cudaSuccess;
}

// Row stride: a half-warp's 8-byte accesses cover eight strips of two neighbouring
// rows (16 floats each), which start on different banks when the stride is 16
// modulo 32; narrower rows follow each other without a gap.
template <typename T>
int row_stride(int nx, bool twod) {
    if (sizeof(T) != 4 || twod || nx < 16) return nx;
    return nx + ((48 - nx % 32) % 32);
}

}  // namespace

cudaError_t tail_configure() {
    cudaError_t e;
    if ((e = configure_one<float, false>()) != cudaSuccess) return e;
    if ((e = configure_one<float, true>()) != cudaSuccess) return e;
    if ((e = configure_one<double, false>()) != cudaSuccess) return e;
    return configure_one<double, true>();
}

// Layout of levels lv[0 .. nl) (nx, ny, nz set; two-dimensional ones as nx x 1 x ny)
// in the shared memory of a cluster: false where they do not fit.
template <typename T>
bool tail_plan(TailParams<T>& p, bool twod, TailLaunch* out) {
    if (p.nl < 1 || p.nl > kTailMaxLevels) return false;
    const int cap = tail_threads<T>();
    const unsigned sizes = twod ? TailCaps<T, true>::sizes : TailCaps<T, false>::sizes;
    const long long whole = sizeof(T) == 8 ? kTailWhole64 : kTailWhole;
    int nc = 1;
    {
        // the cluster that leaves each CTA the fewest plane pairs of the first level, the
        // smallest such
        const TailLevel<T>& L = p.lv[0];
        const long long cells = (long long)L.nx * L.ny * L.nz;
        if (sizeof(T) == 8 && cells > (p.nl == 1 ? kTailCoarse64 : kTailCells64)) return false;
        const int np = L.nz / 2;
        if (cells > whole)
            for (int n = 2; n <= kTailMaxNC && n <= np; ++n)
                if (((sizes >> n) & 1u) && (np + n - 1) / n < (np + nc - 1) / nc) nc = n;
    }
    size_t words = 0;
    int threads = 32;
    for (int l = 0; l < p.nl; ++l) {
        TailLevel<T>& L = p.lv[l];
        if ((L.nx & 1) || (L.nz & 1) || (!twod && (L.ny & 1)) || L.nx < 2 || L.nz < 2) return false;
        const long long cells = (long long)L.nx * L.ny * L.nz;
        const int np = L.nz / 2;
        const long long per_pair = (long long)(L.nx / 2) * L.ny;
        L.split = (nc > 1 && cells > whole) ? 1 : 0;
        const int pairs = L.split ? (np + nc - 1) / nc : np;
        if (pairs * per_pair > cap) return false;
        const int n = pairs * (int)per_pair;
        threads = std::max(threads, n);
        L.group = L.split || n > kFourWarps ? 0 : (n > 32 ? 1 : 2);
        L.row = row_stride<T>(L.nx, twod);
        L.fld = (2 * pairs + (L.split ? 2 : 0)) * L.row * L.ny;
        L.buf = (int)words;
        words += 2 * (size_t)L.fld;
        L.f = (int)words;
        words += (size_t)2 * pairs * L.nx * L.ny;
        L.scaled = (int)words;                   // (even, as every size before it)
        if (l < p.nl - 1) words += 2 * (size_t)p.s;
        if (words * sizeof(T) > kSmemLimit) return false;
        L.inv_cells = T(1.0 / double(cells));
        L.inv_nq = 1.0f / float(L.nx / 2);
        L.inv_ny = 1.0f / float(L.ny);
        L.inv_pairs = 1.0f / float(np);
        if (L.split)
            for (int r = 0; r <= nc; ++r) L.first[r] = (short)first_pair(r, np, nc);
    }
    threads = (threads + 31) / 32 * 32;
    if (p.loop) {                                // four double2 a thread: phi and r of its cells
        words = (words + 3) / 4 * 4;
        p.resident_off = (int)words;
        words += (size_t)16 * threads;
        if (words * sizeof(T) > kSmemLimit) return false;
    }
    out->nc = nc;
    out->threads = threads;
    out->bytes = words * sizeof(T);
    return true;
}

unsigned tail_wait_failures() {
    unsigned n = 0;
    if (cudaMemcpyFromSymbol(&n, g_tail_wait_timeouts, sizeof(n)) != cudaSuccess) return 0;
    return n;
}

template <typename T>
cudaError_t launch_tail(const TailParams<T>& p, bool twod, const TailLaunch& t, cudaStream_t st) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = tail_config(t.nc, t.threads, t.bytes, st, at);
    return twod ? cudaLaunchKernelEx(&cfg, k_tail_levels<T, true>, p)
                : cudaLaunchKernelEx(&cfg, k_tail_levels<T, false>, p);
}

template bool tail_plan<float>(TailParams<float>&, bool, TailLaunch*);
template bool tail_plan<double>(TailParams<double>&, bool, TailLaunch*);
template cudaError_t launch_tail<float>(const TailParams<float>&, bool, const TailLaunch&, cudaStream_t);
template cudaError_t launch_tail<double>(const TailParams<double>&, bool, const TailLaunch&, cudaStream_t);

}  // namespace sg
