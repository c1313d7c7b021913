// Fused RKL super-step for s = 2 and 3 (App. A, Eq. RKL_intermediate_source) with
// every thread on one column: all stages in one pass over the level, FP32, for the
// error equation of the mixed-precision V-cycle (homogeneous Dirichlet or periodic
// ghosts).  Same arithmetic, strip by strip, as k_superstep_lean: the results are
// equal to the last bit.  Against one launch per stage they differ by FP32 rounding:
// off from 64 bits by 0.91 - 1.01e-7 of the result (RKL2, s = 3, smooth fields), the
// stages by 0.95 - 0.99e-7 (sum_exact in sg_superstep.cuh).
//
// Work split.  A CTA owns a column of tx x ty cells widened by four cells in x and
// s in y, one thread per strip of four x cells, and streams it along z.  In the phase
// that plane t arrives, a thread runs stage 1 on plane t - 1, stage 2 on t - 2 and
// stage 3 on t - 3 of its own strip.  The planes above and below are its own, in
// registers, as are the combined fields W_j that stage 1 hands on; shared memory
// holds only what the neighbours in x and y need: one strip and its two end cells
// per stage and phase, double-buffered, so that one barrier a phase is enough.  The
// halo shrinks by a cell per stage; what a thread computes past it is not used.
//
// What bounds it.  The shared-memory pipe (about 52 wavefronts per warp and phase) and the
// issue of its bursts after each barrier; HBM (Y0, f and Y_s once: 30 us at 256^3) is not.
// One general s = 3 super-step, one stage per thread (k_superstep_lean) and here: 512^3
// 831 and 417 us, 256^3 119 and 70, 192^3 59 and 39, 128^3 28 and 20 (cold L2); Y0 = 0:
// 256^3 70 and 47 us.  What gave how much at 256^3: this split 96 us; constant ring
// slots and buffer halves (phases unrolled by six), coefficients as pairs in the
// constant bank and reflected strips copied like any other 82; f, which no neighbour
// reads, loaded into registers a phase ahead 70.  Row pairs per thread
// (384 threads of 158 registers: fewer wavefronts, too few warps) 94 us, 512 threads
// 100, end cells by shuffles 104.
#include "sg_superstep.cuh"

#include <algorithm>
#include <cstdint>
#include <type_traits>

namespace sg {

namespace {

constexpr int kColThreads = 640;        // 20 warps of up to 96 registers
constexpr int kColRing = 6;             // planes of the copy ring: four in flight ahead of the phase's own

template <int S, bool ZERO, bool VEC>
struct Col {
    static constexpr int NS = ZERO ? S - 1 : S;          // stencil stages (Y0 = 0: stage 1 is a multiple of f)
    static constexpr int NF = ZERO || VEC ? 1 : 2;       // staged fields: f; Y0 (VEC: f goes to registers); Y0 and f
    static constexpr int STRIP = 4 * kColThreads;        // floats of one field's strips
    static constexpr int SLOT = NF * STRIP;
    static constexpr int OE = kColRing * SLOT;           // end cells of the staged plane: 2 x (x, w)
    static constexpr int EDGE = 2 * kColThreads;
    static constexpr int OY = OE + 2 * EDGE;             // Y_j, j < NS: 2 x (strips, end cells)
    static constexpr int YBUF = STRIP + EDGE;
    static constexpr int NFLOATS = OY + (NS - 1) * 2 * YBUF;
    static constexpr size_t BYTES = size_t(NFLOATS) * sizeof(float);
    static_assert(BYTES <= 227u * 1024u, "shared memory of one CTA");
};

// The coefficients of LeanCoef as pairs of equal floats: operands of the packed FP32
// instructions straight from the constant bank.
struct ColCoef {
    FirstCoef first;
    float2 ax[2], ay[2], az[2], b[2];               // stages 2 and 3 (Y0 = 0: Y2 from f, then stage 3)
    float kz3;
};

struct ColPlan {
    int q = 0, h = 0;                   // strips and rows of the widened tile
    int tx = 0, ty = 0, tiles_x = 0, tiles_y = 0, chunks = 0, kchunk = 0, threads = 0;
};


// VEC: rows are whole strips (nx % 4 = 0, aligned arrays).  Every strip is then one
// 16-byte copy: a reflected strip is its mirror image, reversed and negated on landing.
template <int S, bool ZERO, bool VEC>
__global__ void __launch_bounds__(kColThreads, 1)
k_superstep_columns(const __grid_constant__ LevelGeom g, const __grid_constant__ ColCoef k,
                    const __grid_constant__ ColPlan p, const float* __restrict__ y0g, const float* __restrict__ fg,
                    float* __restrict__ outg) {
    using C = Col<S, ZERO, VEC>;
    constexpr int NS = C::NS, R = kColRing;
    extern __shared__ __align__(128) float sm[];
    const int tid = threadIdx.x;
    const int nx = g.nx, ny = g.ny, nz = g.nz, plane = nx * ny;
    const bool pz = g.per[2] != 0;
    const int tile = blockIdx.x / p.chunks, chunk = blockIdx.x % p.chunks;
    const int kz0 = chunk * p.kchunk, kz1 = min(nz, kz0 + p.kchunk);
    const int row = tid / p.q, q = tid % p.q;
    const int gx = (tile % p.tiles_x) * p.tx + 4 * (q - 1), gy = (tile / p.tiles_x) * p.ty + row - NS;

    // source of this thread's strip
    LoadDesc ld;
    ld.dst = -1;
    ld.flags = 0;
    bool some = row < p.h, neg = false, rev = false;
    int off = 0;
    if constexpr (VEC) {
        int sx, sy;
        const int xa = map_axis(gx, nx, g.per[0] != 0, &sx), ya = map_axis(gy, ny, g.per[1] != 0, &sy);
        rev = sx < 0;
        neg = sx * sy < 0;
        off = ya * nx + (rev ? xa - 3 : xa);
    } else if (some) {
        ld = make_desc(4 * tid, gx, gy, g, false);
    }
    const int st_n = min(4, nx - gx);
    const bool stores = row >= NS && row < p.h - NS && q >= 1 && q < p.q - 1 && gy < ny && st_n > 0;
    int out_i = (kz0 - 2 * NS) * plane + gy * nx + gx;      // plane t - NS of phase 0

    // neighbours' strips and end cells (clamped: past the block's ends nothing is used)
    const int iu = max(tid - p.q, 0), id = min(tid + p.q, kColThreads - 1);
    const int il = max(tid - 1, 0), ir = min(tid + 1, kColThreads - 1);
    const float *s_own = sm + 4 * tid, *s_up = sm + 4 * iu, *s_dn = sm + 4 * id;
    const float *e_l = sm + kColThreads + il, *e_r = sm + ir;
    float *w_own = sm + 4 * tid, *w_end = sm + tid;

    const int t0 = kz0 - NS;                        // first staged plane
    const int nph = kz1 - kz0 + 2 * NS;             // phases = staged planes
    auto stage_plane = [&](int v, int slot) {
        int zsign;
        const int src = map_axis(t0 + v, nz, pz, &zsign) * plane;
        float* dst = sm + slot * C::SLOT;
        if constexpr (VEC) {
            if (some) {
                cpa16(dst + 4 * tid, (ZERO ? fg : y0g) + (src + off));
            }
        } else {
            if constexpr (!ZERO) issue(ld, dst, y0g + src);
            issue(ld, dst + (C::NF - 1) * C::STRIP, fg + src);
        }
    };
#pragma unroll
    for (int v = 0; v < R - 2; ++v) {
        if (v < nph) stage_plane(v, v);
        cpa_commit();
    }

    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    struct Nb {
        float4 n, s;
        float l, r;
    };
    // what a strip needs from the plane whose strips start at word `strips` and end cells at `ends`
    auto around = [&](int strips, int ends) {
        return Nb{ld4(s_up + strips), ld4(s_dn + strips), e_l[ends], e_r[ends]};
    };
    auto publish_ends = [&](int ends, const float4& v) {
        w_end[ends] = v.x;
        w_end[ends + kColThreads] = v.w;
    };

    float4 f_next = zero4;
    bool ng_before = false;
    // Phase u, u % 6 = U: the z windows, the W fields, the ring slots and the halves of the
    // buffers rotate by constants (a: the staged field, b and c: the outputs of the first two
    // stencil stages)
    auto phase = [&](auto Uc, int u, const float4& a_dn, const float4& a_cn, float4& a_up, const float4& b_dn,
                     const float4& b_cn, float4& b_up, const float4& c_dn, const float4& c_cn, float4& c_up,
                     const float4& w2r, float4& w2w, const float4& w3r, float4& w3w) {
        constexpr int U = decltype(Uc)::value, par = U & 1;
        constexpr int now = U * C::SLOT, before = (U + R - 1) % R * C::SLOT;
        constexpr int eb = C::OE + (par ^ 1) * C::EDGE;
        [[maybe_unused]] constexpr int yb = C::OY + (par ^ 1) * C::YBUF;
        // plane t has landed (this thread's copies): turn its reflected cells
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kColRing - 3) : "memory");
        int zsign = 1;
        const int zt = map_axis(t0 + u, nz, pz, &zsign);
        a_up = ld4(s_own + now);
        [[maybe_unused]] float4 f = f_next;         // f of plane t - 1, loaded a phase ago
        if constexpr (VEC) {
            if (!ZERO && some) f_next = __ldg(reinterpret_cast<const float4*>(fg + (zt * plane + off)));
            auto turn = [&](float4 v, bool ng) {
                if (rev) v = make_float4(v.w, v.z, v.y, v.x);
                return ng ? make_float4(-v.x, -v.y, -v.z, -v.w) : v;
            };
            const bool ng = neg != (zsign < 0);
            if (!ZERO && (rev || ng_before)) f = turn(f, ng_before);
            if (rev || ng) {
                a_up = turn(a_up, ng);
                st4(w_own + now, a_up);
            }
            ng_before = ng;
        } else {
            fixup(ld, sm + now, zsign);
            if constexpr (!ZERO) fixup(ld, sm + now + C::STRIP, zsign);
            a_up = ld4(s_own + now);
        }

        const Nb e1 = around(before, eb);
        float4 v;
        if constexpr (ZERO) {
            v = later_strip(a_cn, e1.n, e1.s, a_dn, a_up, e1.l, e1.r, k.ax[0], k.ay[0], k.az[0], k.b[0], zero4);
            if constexpr (NS >= 2) {
                b_up = v;
                const Nb e2 = around(yb, yb + C::STRIP);
                v = later_strip(b_cn, e2.n, e2.s, b_dn, b_up, e2.l, e2.r, k.ax[1], k.ay[1], k.az[1], k.b[1],
                                scale4(k.kz3, a_dn));
            }
        } else {
            if constexpr (!VEC) f = ld4(s_own + before + C::STRIP);
            first_strip<S>(k.first, a_cn, e1.n, e1.s, a_dn, a_up, e1.l, e1.r, f, b_up, w2w, w3w);
            const Nb e2 = around(yb, yb + C::STRIP);
            v = later_strip(b_cn, e2.n, e2.s, b_dn, b_up, e2.l, e2.r, k.ax[0], k.ay[0], k.az[0], k.b[0], w2r);
            if constexpr (S == 3) {
                c_up = v;
                constexpr int cb = yb + 2 * C::YBUF;
                const Nb e3 = around(cb, cb + C::STRIP);
                v = later_strip(c_cn, e3.n, e3.s, c_dn, c_up, e3.l, e3.r, k.ax[1], k.ay[1], k.az[1], k.b[1], w3r);
            }
        }
        if (stores && u >= 2 * NS) store_out(outg + out_i, v, VEC, st_n);
        out_i += plane;

        publish_ends(C::OE + par * C::EDGE, a_up);
        if constexpr (NS >= 2) {
            constexpr int y = C::OY + par * C::YBUF;
            st4(w_own + y, b_up);
            publish_ends(y + C::STRIP, b_up);
        }
        if constexpr (NS >= 3) {
            constexpr int y = C::OY + (2 + par) * C::YBUF;
            st4(w_own + y, c_up);
            publish_ends(y + C::STRIP, c_up);
        }
        // plane t + R - 2 into the slot of plane t - 2, whose last readers passed the previous barrier
        if (u + R - 2 < nph) stage_plane(u + R - 2, (U + R - 2) % R);
        cpa_commit();
        __syncthreads();
    };

    float4 a0 = zero4, a1 = zero4, a2 = zero4, b0 = zero4, b1 = zero4, b2 = zero4, c0 = zero4, c1 = zero4, c2 = zero4;
    float4 w20 = zero4, w21 = zero4, w22 = zero4, w30 = zero4, w31 = zero4, w32 = zero4;
    auto three = [&](auto Uc, int u) -> bool {      // false: the last phase is done (nph is uniform)
        constexpr int U = decltype(Uc)::value;
        phase(std::integral_constant<int, U>{}, u, a1, a2, a0, b1, b2, b0, c1, c2, c0, w22, w20, w31, w30);
        if (u + 1 >= nph) return false;
        phase(std::integral_constant<int, U + 1>{}, u + 1, a2, a0, a1, b2, b0, b1, c2, c0, c1, w20, w21, w32, w31);
        if (u + 2 >= nph) return false;
        phase(std::integral_constant<int, U + 2>{}, u + 2, a0, a1, a2, b0, b1, b2, c0, c1, c2, w21, w22, w30, w32);
        return u + 3 < nph;
    };
    for (int u = 0; three(std::integral_constant<int, 0>{}, u) && three(std::integral_constant<int, 3>{}, u + 3); u += 6) {}
}

int g_col_sms = 152;

// The cheapest launch: tiles of equal widths and rows that fit one block, z in equal
// chunks; the time of a launch is taken as its waves x phases x (warps + a phase's
// fixed part).  Against up to 26 other plans of a level, 48 x 40 x 56 to 192^3, it came
// within a timer step (2 us) of the best in all but one of 21.
ColPlan col_plan(const LevelGeom& g, int ns) {
    ColPlan best;
    double best_cost = 1e300;
    for (int gx = 1; gx <= (g.nx + 3) / 4; ++gx) {
        const int tx = ((g.nx + gx - 1) / gx + 3) / 4 * 4, q = tx / 4 + 2;
        const int rows = kColThreads / q - 2 * ns;
        if (rows < 1) continue;
        if ((g.nx + tx - 1) / tx != gx) continue;
        const int gy0 = (g.ny + rows - 1) / rows;
        for (int gy = gy0; gy <= std::min(g.ny, gy0 + 3); ++gy) {
            const int ty = (g.ny + gy - 1) / gy, h = ty + 2 * ns;
            if ((g.ny + ty - 1) / ty != gy) continue;
            const int warps = (q * h + 31) / 32;
            const long long tiles = (long long)gx * gy;
            for (int w = 1; w <= 3; ++w) {          // chunks that fill w waves
                const long long c = std::min<long long>(g.nz, std::max(1LL, w * (long long)g_col_sms / tiles));
                const int kchunk = (int)((g.nz + c - 1) / c), chunks = (g.nz + kchunk - 1) / kchunk;
                const long long waves = (tiles * chunks + g_col_sms - 1) / g_col_sms;
                const double cost = double(waves) * (kchunk + 2 * ns + 2) * (6 + warps);
                if (cost < best_cost) {
                    best_cost = cost;
                    best.q = q;
                    best.h = h;
                    best.tx = tx;
                    best.ty = ty;
                    best.tiles_x = gx;
                    best.tiles_y = gy;
                    best.chunks = chunks;
                    best.kchunk = kchunk;
                    best.threads = 32 * warps;
                }
            }
        }
        if (tx <= 32) break;                        // narrower tiles are mostly halo
    }
    return best;
}

ColCoef col_coef(const LeanCoef& k, bool zero) {
    auto two = [](float v) { return make_float2(v, v); };
    ColCoef c{};
    c.first = first_coef(k);
    c.ax[0] = two(zero ? k.zx : k.ax[2]);
    c.ay[0] = two(zero ? k.zy : k.ay[2]);
    c.az[0] = two(zero ? k.zz : k.az[2]);
    c.b[0] = two(zero ? k.zb : k.b[2]);
    c.ax[1] = two(k.ax[3]);
    c.ay[1] = two(k.ay[3]);
    c.az[1] = two(k.az[3]);
    c.b[1] = two(k.b[3]);
    c.kz3 = k.kz[3];
    return c;
}

template <int S, bool ZERO>
cudaError_t col_run(const LevelGeom& g, const ColCoef& k, const float* y0, const float* f, float* out,
                    cudaStream_t st) {
    using C = Col<S, ZERO, false>;
    const bool aligned = ((reinterpret_cast<uintptr_t>(y0) | reinterpret_cast<uintptr_t>(f) |
                           reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const ColPlan p = col_plan(g, C::NS);
    const unsigned grid = (unsigned)(p.tiles_x * p.tiles_y * p.chunks);
    if ((g.nx & 3) == 0 && aligned) k_superstep_columns<S, ZERO, true><<<grid, p.threads, Col<S, ZERO, true>::BYTES, st>>>(g, k, p, y0, f, out);
    else k_superstep_columns<S, ZERO, false><<<grid, p.threads, C::BYTES, st>>>(g, k, p, y0, f, out);
    return cudaGetLastError();
}

template <int S, bool ZERO>
cudaError_t col_configure() {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(k_superstep_columns<S, ZERO, true>, attr, (int)Col<S, ZERO, true>::BYTES);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_superstep_columns<S, ZERO, false>, attr, (int)Col<S, ZERO, false>::BYTES);
}

}  // namespace

cudaError_t columns_configure() {
    cudaError_t e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&g_col_sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = col_configure<2, false>()) != cudaSuccess) return e;
    if ((e = col_configure<2, true>()) != cudaSuccess) return e;
    if ((e = col_configure<3, false>()) != cudaSuccess) return e;
    return col_configure<3, true>();
}

// (by the attribute that columns_configure sets last)
bool columns_configured() {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, k_superstep_columns<3, true, false>) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.maxDynamicSharedSizeBytes == (int)Col<3, true, false>::BYTES;
}

cudaError_t launch_superstep_columns(const LevelGeom& g, int order, int s, bool zero_y0, const FusedCoef& cf,
                                     const float* y0, const float* f, float* out, cudaStream_t st) {
    const ColCoef k = col_coef(make_lean_coef(g, order, s, cf), zero_y0);
    if (s == 2) return zero_y0 ? col_run<2, true>(g, k, y0, f, out, st) : col_run<2, false>(g, k, y0, f, out, st);
    if (s == 3) return zero_y0 ? col_run<3, true>(g, k, y0, f, out, st) : col_run<3, false>(g, k, y0, f, out, st);
    return cudaErrorInvalidValue;
}

}  // namespace sg
