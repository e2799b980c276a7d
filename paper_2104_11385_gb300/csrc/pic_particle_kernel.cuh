// pic_particle_kernel.cuh -- the particle side of the PIC cycle on sm_103a,
// templated on the arithmetic of the particle push (included by one
// translation unit per precision and dimensionality:
// pic_particles_{f64,f32}_{3d,2d}.cu).
//
// pic_particle_kernel: persistent CTAs pull work units (a chunk of one box's
// particles) from cost-ordered lists.  For every tile (sub-box) a unit touches,
// the guard-extended E/B tile is staged into shared memory by TMA
// (cp.async.bulk.tensor, local HBM only, no multicast).  The current goes
// straight into the guard-padded global J arrays as fire-and-forget FP64
// reductions (red.global.add.f64, performed in L2) in every precision, and the
// particle loads are staged through shared memory with cp.async one loop
// iteration ahead.
//
// What bounds it (FP64, linear, 128^3 foil, 8.4 M particles): the FP64 pipe
// takes one warp instruction per SM every 16 clocks, and a particle's gather,
// push and deposit are 165 FP64 instructions, 2.73 ms at 86 % of that pipe.
// The gather (60 of them) and the deposit (36) run in 64-bit fixed point on the
// integer pipes instead (pic_fix.cuh), the Boris push keeps 51: 1.40 ms, 2717
// issued instructions per 32 particles, issue slots 43 % and FP64 pipe 56 % busy
// (16 warps per SM by registers: latency-bound between the two).  Each thread
// brackets its particle loop with clock64(); the deltas are warp-reduced, summed in shared memory and
// added once per unit to the box's cost -- the device-clock cost of
// arXiv 2104.11385 Sec. 2.2 (Fig. 2a); thread 0 adds the %globaltimer span
// of the unit's particle loops, averaged over the warps, to the box's
// kernel-time cost.  The same pass writes each particle's new
// tile key and the per-tile histogram for the re-sort.
//
// Physics per particle (the schemes the paper leaves open, Sec. 2.1): field
// gather with B-spline shapes of order 1-3 at each component's Yee location
// (same order in every direction, or the energy-conserving variant with one
// order less along the staggered directions), relativistic Boris push,
// Esirkepov charge-conserving deposit (Esirkepov 2001).  The cost capture can
// be switched off per simulation to measure its overhead.
#pragma once
#include <type_traits>

#include "pic_arith.cuh"
#include "pic_fix.cuh"
#include "pic_internal.h"
#include "pic_sync.cuh"

namespace {

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Exact floor and fractional part of x.  On GB300 every FP64 instruction,
// conversions included, issues at the FP64 rate (about 2 per SM per clock), so
// for 0 <= x < 2^31 both come from integer work on the IEEE-754 bits; other x
// go through floor().  Both routes give the identical (exact) results.  The
// floor() route is a separate function: inlined, the compiler predicates it,
// and its FP64 instructions then occupy the FP64 pipe on every call.
struct IFrac {
    int i;
    double f;
};
static __device__ __noinline__ IFrac ifloor_frac_slow(double x) {
    const double fl = floor(x);
    return IFrac{(int)fl, x - fl};
}
static __device__ __noinline__ int ifloor_slow(double x) { return (int)floor(x); }

__device__ __forceinline__ int ifloor_frac(double x, double& f) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((unsigned long long)b >> 52) - 1023;  // sign set -> e > 1023
    if (e < 0) {
        if (b >= 0) {  // 0 <= x < 1
            f = x;
            return 0;
        }
    } else if (e < 31) {
        const unsigned long long m = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
        const int sh = 52 - e;
        const int i = (int)(m >> sh);
        const unsigned long long fm = m & ((1ull << sh) - 1ull);
        if (fm == 0ull) {
            f = 0.0;
        } else {
            const int top = 63 - __clzll((long long)fm);
            const unsigned long long bits = ((unsigned long long)(top - sh + 1023) << 52) |
                                            ((fm << (52 - top)) & 0xFFFFFFFFFFFFFull);
            f = __longlong_as_double((long long)bits);
        }
        return i;
    }
    const IFrac r = ifloor_frac_slow(x);
    f = r.f;
    return r.i;
}

// floor of x >= 0 (x < 2^31) by integer work; floor() otherwise
__device__ __forceinline__ int ifloor(double x) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((unsigned long long)b >> 52) - 1023;
    if (e < 0 && b >= 0) return 0;
    if (e >= 0 && e < 31)
        return (int)((((unsigned long long)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) >> (52 - e));
    return ifloor_slow(x);
}

// periodic image of a position that left [0, n) by less than n: a separate
// function, so that the rare FP64 add is a branch and not a predicated
// instruction holding the FP64 pipe for every particle
static __device__ __noinline__ double wrap_periodic(double x, double n) { return x < 0.0 ? x + n : x - n; }

// x < 0 and x >= y for y > 0 by integer comparison of the bit patterns
__device__ __forceinline__ bool is_neg(double x) { return __double_as_longlong(x) < 0; }
__device__ __forceinline__ bool ge_pos(double x, double y) {
    return __double_as_longlong(x) >= __double_as_longlong(y);
}
__device__ __forceinline__ bool ge_half(double f) {  // f >= 0.5 for f >= 0
    return __double_as_longlong(f) >= 0x3FE0000000000000ll;
}

// one-dimensional B-spline support: first node and ORDER+1 weights in the
// arithmetic type R (double, or float for the FP32 variant)
template <int ORDER, class R>
struct Support {
    int s;
    R w[ORDER + 1];
};

// cubic B-spline weights of the four nodes floor(xi)-1 .. floor(xi)+2, f = frac(xi)
template <class R>
__device__ __forceinline__ void cubic_weights(R f, R* w) {
    using A = Arith<R>;
    const R k6 = A::c(1.0 / 6.0), k23 = A::c(2.0 / 3.0), half = A::c(0.5);
    const R g = A::c(1.0) - f;
    const R f2 = f * f, g2 = g * g;
    w[0] = (g2 * g) * k6;
    w[1] = fma(half * f, f2, k23 - f2);
    w[2] = fma(half * g, g2, k23 - g2);
    w[3] = (f2 * f) * k6;
}

// support of a node-centred quantity at xi (cells, from the tile origin)
template <int ORDER, class R>
__device__ __forceinline__ Support<ORDER, R> support(double xi) {
    using A = Arith<R>;
    Support<ORDER, R> r;
    double f;
    const int i = ifloor_frac(xi, f);
    if constexpr (ORDER == 1) {
        r.s = i;
        const R fr = A::from(f);
        r.w[0] = A::c(1.0) - fr;
        r.w[1] = fr;
    } else if constexpr (ORDER == 2) {
        // nearest node c = floor(xi + 1/2), d = xi - c in [-1/2, 1/2)
        const bool up = ge_half(f);
        const R fr = A::from(f);
        const R d = up ? fr - A::c(1.0) : fr;
        const R a = A::c(0.5) - d, b = A::c(0.5) + d;
        r.s = i + (up ? 1 : 0) - 1;
        r.w[0] = A::c(0.5) * (a * a);
        r.w[1] = fma(-d, d, A::c(0.75));
        r.w[2] = A::c(0.5) * (b * b);
    } else {
        r.s = i - 1;
        cubic_weights<R>(A::from(f), r.w);
    }
    return r;
}

// node and half-node supports of one position (the half-node grid is shifted
// by +1/2 cell: Ex along x, etc.), and the cell floor(xi).  ec selects the
// energy-conserving half-node support: order ORDER - 1 (order 0: the nearest
// half node), stored with a zero last weight so that the interpolation code
// is shared.
template <int ORDER, class R>
__device__ __forceinline__ void supports(double xi, bool ec, Support<ORDER, R>& nd, Support<ORDER, R>& hf,
                                         int& cell) {
    using A = Arith<R>;
    double f;
    const int i = ifloor_frac(xi, f);
    cell = i;
    const bool up = ge_half(f);
    const R fr = A::from(f);
    if constexpr (ORDER == 1) {
        nd.s = i;
        nd.w[0] = A::c(1.0) - fr;
        nd.w[1] = fr;
        if (ec) {  // box shape: half node i (at i + 1/2) carries the point
            hf.s = i;
            hf.w[0] = A::c(1.0);
            hf.w[1] = A::c(0.0);
        } else {
            const R g = fr + (up ? A::c(-0.5) : A::c(0.5));  // xi - 1/2 - floor(xi - 1/2)
            hf.s = up ? i : i - 1;
            hf.w[0] = A::c(1.0) - g;
            hf.w[1] = g;
        }
    } else if constexpr (ORDER == 2) {
        const R d = up ? fr - A::c(1.0) : fr;  // node: xi - floor(xi + 1/2)
        const R a = A::c(0.5) - d, b = A::c(0.5) + d;
        nd.s = i + (up ? 1 : 0) - 1;
        nd.w[0] = A::c(0.5) * (a * a);
        nd.w[1] = fma(-d, d, A::c(0.75));
        nd.w[2] = A::c(0.5) * (b * b);
        if (ec) {  // hat on the half-node grid: g = frac(xi - 1/2)
            const R g = fr + (up ? A::c(-0.5) : A::c(0.5));
            hf.s = up ? i : i - 1;
            hf.w[0] = A::c(1.0) - g;
            hf.w[1] = g;
            hf.w[2] = A::c(0.0);
        } else {
            const R h = fr - A::c(0.5);  // half: (xi - 1/2) - floor(xi), nearest half-node floor(xi)
            const R ah = A::c(0.5) - h, bh = A::c(0.5) + h;
            hf.s = i - 1;
            hf.w[0] = A::c(0.5) * (ah * ah);
            hf.w[1] = fma(-h, h, A::c(0.75));
            hf.w[2] = A::c(0.5) * (bh * bh);
        }
    } else {
        nd.s = i - 1;
        cubic_weights<R>(fr, nd.w);
        if (ec) {  // quadratic on the half-node grid around the nearest half node floor(xi)
            const R h = fr - A::c(0.5);
            const R ah = A::c(0.5) - h, bh = A::c(0.5) + h;
            hf.s = i - 1;
            hf.w[0] = A::c(0.5) * (ah * ah);
            hf.w[1] = fma(-h, h, A::c(0.75));
            hf.w[2] = A::c(0.5) * (bh * bh);
            hf.w[3] = A::c(0.0);
        } else {
            const R g = fr + (up ? A::c(-0.5) : A::c(0.5));
            hf.s = (up ? i : i - 1) - 1;
            cubic_weights<R>(g, hf.w);
        }
    }
}

// supports relative to a tile origin o, from the global position: floor and
// fraction of x are those of x - o (o an integer), without forming x - o
template <int ORDER, class R>
__device__ __forceinline__ Support<ORDER, R> support_at(double x, int o) {
    Support<ORDER, R> r = support<ORDER, R>(x);
    r.s -= o;
    return r;
}
template <int ORDER, class R>
__device__ __forceinline__ void supports_at(double x, int o, bool ec, Support<ORDER, R>& nd,
                                            Support<ORDER, R>& hf, int& cell) {
    supports<ORDER, R>(x, ec, nd, hf, cell);
    nd.s -= o;
    hf.s -= o;
    cell -= o;
}

// E/B tile halo below the tile origin: 1 cell (orders 1, 2), 2 cells (order 3)
template <int ORDER>
struct EBHalo {
    static constexpr int lo = ORDER == 3 ? 2 : 1;
};

// interpolation of one component from R values with extents (SX, SY): a shared
// tile (FP32), or in FP64 the global arrays (I = int64_t)
template <class R, int ORDER, int DIM, class I>
__device__ __forceinline__ R interp(const R* __restrict__ F, I SX, I SY, const Support<ORDER, R>& sx,
                                    const Support<ORDER, R>& sy, const Support<ORDER, R>& sz) {
    // tile column 0 is local cell -EBHalo<ORDER>::lo
    constexpr int H = EBHalo<ORDER>::lo;
    if constexpr (ORDER == 1) {
        // linear: nested lerps a + f (b - a) need only the fractional parts
        auto lerp = [](R a, R b, R f) { return fma(f, b - a, a); };
        const R fx = sx.w[1];
        if constexpr (DIM == 3) {
            const R* r00 = F + ((sz.s + H) * SY + (sy.s + H)) * SX + (sx.s + H);
            const R* r10 = r00 + SX;
            const R* r01 = r00 + SX * SY;
            const R* r11 = r01 + SX;
            const R a0 = lerp(lerp(r00[0], r00[1], fx), lerp(r10[0], r10[1], fx), sy.w[1]);
            const R a1 = lerp(lerp(r01[0], r01[1], fx), lerp(r11[0], r11[1], fx), sy.w[1]);
            return lerp(a0, a1, sz.w[1]);
        } else {
            const R* r0 = F + (sz.s + H) * SX + (sx.s + H);
            const R* r1 = r0 + SX;
            return lerp(lerp(r0[0], r0[1], fx), lerp(r1[0], r1[1], fx), sz.w[1]);
        }
    } else if constexpr (DIM == 3) {
        R acc;
#pragma unroll
        for (int c = 0; c <= ORDER; ++c) {
            R pl;
#pragma unroll
            for (int b = 0; b <= ORDER; ++b) {
                const R* row = F + ((sz.s + H + c) * SY + (sy.s + H + b)) * SX + (sx.s + H);
                R r = sx.w[0] * row[0];
#pragma unroll
                for (int a = 1; a <= ORDER; ++a) r = fma(sx.w[a], row[a], r);
                pl = (b == 0) ? sy.w[0] * r : fma(sy.w[b], r, pl);
            }
            acc = (c == 0) ? sz.w[0] * pl : fma(sz.w[c], pl, acc);
        }
        return acc;
    } else {
        R acc;
#pragma unroll
        for (int c = 0; c <= ORDER; ++c) {
            const R* row = F + (sz.s + H + c) * SX + (sx.s + H);
            R r = sx.w[0] * row[0];
#pragma unroll
            for (int a = 1; a <= ORDER; ++a) r = fma(sx.w[a], row[a], r);
            acc = (c == 0) ? sz.w[0] * r : fma(sz.w[c], r, acc);
        }
        return acc;
    }
}

// The six E/B components at one particle.  E_a sits on the half-node grid
// along a and on nodes across it, B_a the other way round.
template <class R, int ORDER, int DIM>
__device__ __forceinline__ void gather6(const R* __restrict__ sEB, int stride, int SX, int SY,
                                        const Support<ORDER, R>* nd, const Support<ORDER, R>* hf, R* e,
                                        R* b) {
    e[0] = interp<R, ORDER, DIM>(sEB, SX, SY, hf[0], nd[1], nd[2]);
    e[1] = interp<R, ORDER, DIM>(sEB + stride, SX, SY, nd[0], hf[1], nd[2]);
    e[2] = interp<R, ORDER, DIM>(sEB + 2 * stride, SX, SY, nd[0], nd[1], hf[2]);
    b[0] = interp<R, ORDER, DIM>(sEB + 3 * stride, SX, SY, nd[0], hf[1], hf[2]);
    b[1] = interp<R, ORDER, DIM>(sEB + 4 * stride, SX, SY, hf[0], nd[1], hf[2]);
    b[2] = interp<R, ORDER, DIM>(sEB + 5 * stride, SX, SY, hf[0], hf[1], nd[2]);
}

template <class T>
__device__ __forceinline__ T pick3(int a, const T& v0, const T& v1, const T& v2) {
    return a == 0 ? v0 : (a == 1 ? v1 : v2);
}

// ---- FP64: fixed-point gather -----------------------------
struct Six {
    double v[6];  // Ex Ey Ez Bx By Bz
};

// the six components from the tile in fixed point (component c at c * stride,
// the biased exponent of its largest magnitude in emax[c]).  Linear shapes
// unroll the six interpolations; the others run them as a loop (27 or 64
// products each: six copies would not fit the instruction cache).
template <int ORDER, int DIM>
__device__ __forceinline__ Six gather6_q(const long long* __restrict__ F, int stride, int SX, int SY,
                                         const int* __restrict__ emax, const AxisQ<ORDER>* nd,
                                         const AxisQ<ORDER>* hf) {
    constexpr int H = EBHalo<ORDER>::lo;
    constexpr int B = 63 - TileBits<ORDER>::FB;  
    Six r;
    if constexpr (ORDER == 1) {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const int a = c < 3 ? c : c - 3;
            const bool isb = c >= 3;
            r.v[c] = fix_double(interp_q<ORDER, DIM, H>(F + c * stride, SX, SY, (a == 0) != isb ? hf[0] : nd[0],
                                                        (a == 1) != isb ? hf[1] : nd[1],
                                                        (a == 2) != isb ? hf[2] : nd[2]),
                                emax[c] + B);
        }
    } else {
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0, v4 = 0.0, v5 = 0.0;
#pragma unroll 1
        for (int c = 0; c < 6; ++c) {
            const int a = c < 3 ? c : c - 3;
            const bool isb = c >= 3;
            const AxisQ<ORDER> sx = ((a == 0) != isb) ? hf[0] : nd[0];
            const AxisQ<ORDER> sy = ((a == 1) != isb) ? hf[1] : nd[1];
            const AxisQ<ORDER> sz = ((a == 2) != isb) ? hf[2] : nd[2];
            const double v = fix_double(interp_q<ORDER, DIM, H>(F + c * stride, SX, SY, sx, sy, sz), emax[c] + B);
            v0 = c == 0 ? v : v0;
            v1 = c == 1 ? v : v1;
            v2 = c == 2 ? v : v2;
            v3 = c == 3 ? v : v3;
            v4 = c == 4 ? v : v4;
            v5 = c == 5 ? v : v5;
        }
        r = Six{{v0, v1, v2, v3, v4, v5}};
    }
    return r;
}

// Component c in FP64 from the global arrays (which the kernel only reads), out of
// line: Inf, NaN, and magnitudes outside the fixed-point exponent range.
template <int ORDER, int DIM>
static __device__ __noinline__ double gather1_fp64(const SimDev& S, int c, double X, double Y, double Z, int ox, int oy,
                                                   int oz) {
    constexpr int H = EBHalo<ORDER>::lo;
    const bool ec = S.ec != 0, isb = c >= 3;
    const int a = isb ? c - 3 : c;
    auto one = [&](double x, int o, bool half) {
        Support<ORDER, double> nd, hf;
        int cell;
        supports_at<ORDER, double>(x, o, ec, nd, hf, cell);
        return half ? hf : nd;
    };
    const Support<ORDER, double> sx = one(X, ox, (a == 0) != isb), sz = one(Z, oz, (a == 2) != isb);
    Support<ORDER, double> sy = sx;
    if (DIM == 3) sy = one(Y, oy, (a == 1) != isb);
    const double* F = S.F[c] + pidx(S, ox - H, DIM == 3 ? oy - H : 0, oz - H);
    if constexpr (ORDER == 1) {
        return interp<double, ORDER, DIM, int64_t>(F, S.pn[0], S.pn[1], sx, sy, sz);
    } else {
        // rolled, few registers: what a call clobbers is spilled around it on the
        // caller's fast path too (unrolled, the cubic kernel spills 500 bytes)
        double v = 0.0;
#pragma unroll 1
        for (int k = 0; k <= ORDER; ++k) {
            double pl = 0.0;
#pragma unroll 1
            for (int j = 0; j <= (DIM == 3 ? ORDER : 0); ++j) {
                const double* row =
                    F + ((sz.s + H + k) * (int64_t)S.pn[1] + (DIM == 3 ? sy.s + H + j : 0)) * S.pn[0] + sx.s + H;
                double l = 0.0;
#pragma unroll
                for (int i = 0; i <= ORDER; ++i) l = fma(sx.w[i], row[i], l);
                pl = DIM == 3 ? fma(sy.w[j], l, pl) : l;
            }
            v = fma(sz.w[k], pl, v);
        }
        return v;
    }
}

// Component c in fixed point from the global arrays, in units of the largest
// magnitude of the particle's own nodes, out of line: for particles where the
// component is marked as weak against its tile's largest.  In FP64 it would hold
// that pipe for 13 instructions of 16 clocks (linear 3D; cubic about 100) against
// about 230 (1000) integer ones at a quarter of a clock.  The first steps of the 2D
// cubic disk at 960^2 cells from zero fields, where noise fields span many
// binades: 4.35 ms per step (in FP64 5.1; with the bits lost 3.4); all components of
// a particle in one call: the same.  Rolled for long shapes, few registers: what a
// call clobbers is spilled around it on the caller's fast path too.
template <int ORDER, int DIM>
static __device__ __noinline__ double gather1_weak(const SimDev& S, int c, double X, double Y, double Z, int ox, int oy,
                                                   int oz) {
    constexpr int FB = TileBits<ORDER>::FB, NY = DIM == 3 ? ORDER : 0;
    const bool ec = S.ec != 0, isb = c >= 3;
    const int a = isb ? c - 3 : c;
    auto axis = [&](double x, int o, bool half) {
        const CellQ q = cell_q(x);
        const SupQ<ORDER> n = node_support<ORDER>(q, o), h = half_support<ORDER>(q, o, ec);
        return axis_of<ORDER>(half ? h : n);
    };
    const AxisQ<ORDER> sx = axis(X, ox, (a == 0) != isb), sz = axis(Z, oz, (a == 2) != isb);
    AxisQ<ORDER> sy = sx;
    if (DIM == 3) sy = axis(Y, oy, (a == 1) != isb);
    const double* const F = S.F[c] + pidx(S, ox + sx.s, DIM == 3 ? oy + sy.s : 0, oz + sz.s);
    const int64_t px = S.pn[0], pxy = px * S.pn[1];
    constexpr int U = ORDER == 1 ? 2 : 1;
    unsigned m = 0u;
#pragma unroll U
    for (int k = 0; k <= ORDER; ++k)
#pragma unroll U
        for (int j = 0; j <= NY; ++j)
#pragma unroll
            for (int i = 0; i <= ORDER; ++i)
                m = max(m, (unsigned)__double2hiint(F[k * pxy + j * px + i]) & 0x7FFFFFFFu);
    const int em = (int)(m >> 20);
    if (em < 128 || !tile_exp_ok(em)) return gather1_fp64<ORDER, DIM>(S, c, X, Y, Z, ox, oy, oz);
    auto at = [&](int k, int j, int i) { return tile_fix<FB>(F[k * pxy + j * px + i], em); };
    long long r;
    if constexpr (ORDER == 1) {
        auto row = [&](int k, int j) { return lerpq(at(k, j, 0), at(k, j, 1), sx.w[1]); };
        if constexpr (DIM == 3)
            r = lerpq(lerpq(row(0, 0), row(0, 1), sy.w[1]), lerpq(row(1, 0), row(1, 1), sy.w[1]), sz.w[1]);
        else
            r = lerpq(row(0, 0), row(1, 0), sz.w[1]);
    } else {
        AccQ vol;
#pragma unroll 1
        for (int k = 0; k <= ORDER; ++k) {
            AccQ pl;
#pragma unroll 1
            for (int j = 0; j <= NY; ++j) {
                AccQ line;
#pragma unroll
                for (int i = 0; i <= ORDER; ++i) line.mac(at(k, j, i), sx.w[i]);
                if constexpr (DIM == 3) pl.mac(line.get(), sy.w[j]);
                else vol.mac(line.get(), sz.w[k]);
            }
            if constexpr (DIM == 3) vol.mac(pl.get(), sz.w[k]);
        }
        r = vol.get();
    }
    return fix_double(r, em + 63 - FB);
}

// Scans a staged tile: emax, the biased exponent of each component's largest
// magnitude, and emin, that of the weakest two neighbours along x that are not both
// zero (of the weakest single element where windows of mark_weak have single nodes
// along x).  No window is weaker than that, so most tiles need no marks.  Elements
// are taken in a row, 62 per warp and round, two per lane from a 16-byte load.
template <int ORDER>
__device__ __forceinline__ void scan_tile(const double* __restrict__ sEB, int stride, int vol, bool ec, int* emax, int* emin) {
    const int lane = threadIdx.x & 31;
    const bool one = ORDER == 1 && ec;
    unsigned mx[6], mn[6];  // high words, the smallest less one (zero becomes the largest)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        mx[c] = 0u;
        mn[c] = 0xFFFFFFFFu;
    }
    for (int i0 = 62 * (threadIdx.x >> 5); i0 < vol; i0 += 62 * (blockDim.x >> 5)) {
        const int i = min(i0 + 2 * lane, vol - 2);  // (vol is even: rows have even lengths)
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const uint4 v = *reinterpret_cast<const uint4*>(sEB + c * stride + i);
            const unsigned e = v.y & 0x7FFFFFFFu, o = v.w & 0x7FFFFFFFu, next = __shfl_down_sync(0xffffffffu, e, 1);
            const bool single = one && ((c < 3 ? c == 0 : c != 3));  // half nodes along x
            const unsigned both = max(e, o), across = lane == 31 ? both : max(o, next);
            mx[c] = max(mx[c], both);
            mn[c] = min(mn[c], min((single ? e : both) - 1u, (single ? o : across) - 1u));
        }
    }
    unsigned hi = 0u, lo = 0u;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const unsigned a = __reduce_max_sync(0xffffffffu, mx[c]), b = __reduce_min_sync(0xffffffffu, mn[c]);
        hi = lane == c ? a : hi;
        lo = lane == c ? b : lo;
    }
    if (lane < 6) {
        atomicMax(emax + lane, (int)(hi >> 20));
        atomicMin(emin + lane, lo == 0xFFFFFFFFu ? 0x7FFF : (int)((lo + 1u) >> 20));
    }
}

// Marks where a component of a staged tile is gathered by itself (gather1_weak): one bit of bits + c
// * words for each window of 2 x 2 x 2 nodes (a single node along the half-node
// directions of the energy-conserving linear gather), numbered by the element i of
// its lower corner (mark_bit), set if it does not reach weak_limit and is not all
// zero.  A particle looks at the window in the middle of its support
// (weak_components).  Of a window the two nodes at the lower corner along x are
// looked at, and the two across from them in y and z: a wave that crosses zero has
// one of them off the crossing, random noise marks hardly a window.  Elements are
// taken in a row across row ends, where windows belong to no particle.  A lane
// takes two windows from two 16-byte loads: shared loads are what this costs,
// waiting behind the other CTA's reductions, 1 to 5 us per staged tile, and only
// the tiles where scan_tile leaves it open pay that (particle kernel per step
// without the marks / marked always / where needed: 16^3 plasma 40.0 / 41.9 / 40.3
// us, foil of 32 x 64 x 128 cells and 541 thousand particles 264 / 280 / 263, 128^3
// foil 1402 / 1419 / 1407).
__device__ __forceinline__ int mark_word(int i) { return ((i >> 6) << 1) | (i & 1); }
__device__ __forceinline__ int mark_bit(int i) { return (i >> 1) & 31; }
template <int ORDER, int DIM>
__device__ __forceinline__ bool mark_weak(unsigned* __restrict__ bits, int words, const double* __restrict__ sEB,
                                          int stride, int vol, int SX, int SY, const int* __restrict__ emax, bool ec) {
    const int lane = threadIdx.x & 31, SZ = DIM == 3 ? SX * SY : SX;
    const bool one = ORDER == 1 && ec;
    unsigned lim[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) lim[c] = emax[c] == 0 ? 0u : weak_limit<ORDER>(emax[c]) << 20;
    const int n = vol - 2 - SZ - (DIM == 3 ? SX : 0);  // last pair of windows that lie in the tile
    unsigned any = 0u;
    for (int w = 2 * (threadIdx.x >> 5); w < words; w += 2 * (blockDim.x >> 5)) {
        const int i = min(32 * w + 2 * lane, n);  // (n is even: rows have even lengths)
        uint2 mine = make_uint2(0u, 0u);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const int a = c < 3 ? c : c - 3;
            const bool isb = c >= 3, hx = (a == 0) != isb, hy = (a == 1) != isb, hz = (a == 2) != isb;
            const int d = (DIM == 2 || (one && hy) ? 0 : SX) + (one && hz ? 0 : SZ);
            const uint4 v = *reinterpret_cast<const uint4*>(sEB + c * stride + i);
            const uint4 u = *reinterpret_cast<const uint4*>(sEB + c * stride + i + d);
            unsigned m0 = max(v.y & 0x7FFFFFFFu, u.y & 0x7FFFFFFFu);  // (high words)
            unsigned m1 = max(v.w & 0x7FFFFFFFu, u.w & 0x7FFFFFFFu);
            const unsigned next = __shfl_down_sync(0xffffffffu, m0, 1);
            if (!(one && hx)) {
                m0 = max(m0, m1);
                m1 = lane == 31 ? m1 : max(m1, next);
            }
            const unsigned w0 = __ballot_sync(0xffffffffu, m0 != 0u && m0 < lim[c]);
            const unsigned w1 = __ballot_sync(0xffffffffu, m1 != 0u && m1 < lim[c]);
            any |= w0 | w1;
            if (lane == c) mine = make_uint2(w0, w1);
        }
        if (lane < 6) *reinterpret_cast<uint2*>(bits + lane * words + w) = mine;
    }
    return any != 0u;
}
// the components (bits) that a particle gathers by itself, from its supports and the marks
template <int ORDER, int DIM>
__device__ __forceinline__ unsigned weak_components(const unsigned* __restrict__ bits, int words, int SX, int SY,
                                                    const SupQ<ORDER>* nd, const AxisQ<ORDER>* hf) {
    // lower node of the window along an axis: for quadratic shapes those at the
    // nearest node and half a cell below it lie in every support
    constexpr int H = EBHalo<ORDER>::lo, BN = H + (ORDER == 1 ? 0 : 1), BH = H + (ORDER == 3 ? 1 : 0);
    auto half = [&](int a) { return (ORDER == 2 ? nd[a].s : hf[a].s) + BH; };
    const int SZ = SX * SY, nx = nd[0].s + BN, hx = half(0), nz = (nd[2].s + BN) * SZ, hz = half(2) * SZ;
    const int ny = DIM == 3 ? (nd[1].s + BN) * SX : 0, hy = DIM == 3 ? half(1) * SX : 0;
    unsigned mask = 0u;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int a = c < 3 ? c : c - 3;
        const bool isb = c >= 3;
        const int i = ((a == 0) != isb ? hx : nx) + ((a == 1) != isb ? hy : ny) + ((a == 2) != isb ? hz : nz);
        mask |= ((bits[c * words + mark_word(i)] >> mark_bit(i)) & 1u) << c;
    }
    return mask;
}

// Esirkepov node shapes on a common window of W nodes starting at the lower of
// the two supports: W = ORDER + 1 when the particle keeps its support (the
// in-cell case, most particles), W = ORDER + 2 when it moves to a neighbour.
template <int ORDER, int W, class R>
struct Window {
    int base;
    R S0[W];
    R DS[W];
};

template <int ORDER, int W, class R>
__device__ __forceinline__ bool make_window(const Support<ORDER, R>& a, const Support<ORDER, R>& b,
                                            Window<ORDER, W, R>& win) {
    int base = min(a.s, b.s);
    int oa = a.s - base, ob = b.s - base;
    // unsigned: a cell index saturated by a move of 2^31 cells or more wraps the difference
    if ((unsigned)oa > (unsigned)(W - ORDER - 1) || (unsigned)ob > (unsigned)(W - ORDER - 1)) return false;
    win.base = base;
    const R zero = Arith<R>::c(0.0);
#pragma unroll
    for (int l = 0; l < W; ++l) {
        R s0 = zero, s1 = zero;
#pragma unroll
        for (int k = 0; k <= ORDER; ++k) {
            s0 = (l - oa == k) ? a.w[k] : s0;
            s1 = (l - ob == k) ? b.w[k] : s1;
        }
        win.S0[l] = s0;
        win.DS[l] = s1 - s0;
    }
    return true;
}

struct Tile {
    int sim;
    int t;
    int o[3];  // origin cell
};

__device__ __forceinline__ void tile_origin(const SimDev& S, int t, int o[3]) {
    int b = t / S.tiles_per_box, lt = t - b * S.tiles_per_box;
    int bx = b % S.nb[0], by = (b / S.nb[0]) % S.nb[1], bz = b / (S.nb[0] * S.nb[1]);
    int tx = lt % S.tpb[0], ty = (lt / S.tpb[0]) % S.tpb[1], tz = lt / (S.tpb[0] * S.tpb[1]);
    o[0] = bx * S.bsz[0] + tx * S.T[0];
    o[1] = by * S.bsz[1] + ty * S.T[1];
    o[2] = bz * S.bsz[2] + tz * S.T[2];
}

// tile key of a global cell (box-major numbering); SV: SimDev or HotSim
template <class SV>
__device__ __forceinline__ int tile_key(const SV& S, int ix, int iy, int iz) {
    int bx = ix / S.bsz[0], by = iy / S.bsz[1], bz = iz / S.bsz[2];
    int tx = (ix - bx * S.bsz[0]) / S.T[0];
    int ty = (iy - by * S.bsz[1]) / S.T[1];
    int tz = (iz - bz * S.bsz[2]) / S.T[2];
    int b = (bz * S.nb[1] + by) * S.nb[0] + bx;
    return b * S.tiles_per_box + (tz * S.tpb[1] + ty) * S.tpb[0] + tx;
}

// A tile's key is a sum of one part per direction.  For the staged tile the
// parts of its own position and of the neighbours' on either side (periodic)
// are kept in shared memory, so that a particle that moved by less than a tile
// finds its new key without the nine integer divisions of tile_key.
template <class SV>
__device__ __forceinline__ int key_part(const SV& S, int a, int i) {
    const int n = S.n[a];
    i = i < 0 ? i + n : (i >= n ? i - n : i);
    const int b = i / S.bsz[a], t = (i - b * S.bsz[a]) / S.T[a];
    const int bs = a == 0 ? 1 : (a == 1 ? S.nb[0] : S.nb[0] * S.nb[1]);
    const int ts = a == 0 ? 1 : (a == 1 ? S.tpb[0] : S.tpb[0] * S.tpb[1]);
    return b * bs * S.tiles_per_box + t * ts;
}
// key of the tile that holds the cell at offset r[a] (unwrapped) from the tile's origin; -1: further off
template <int DIM, class SV>
__device__ __forceinline__ int near_key(const SV& S, const int (*nk)[3], const int r[3]) {
    int key = 0;
    bool near = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) continue;
        const int T = S.T[a];
        near = near && r[a] >= -T && r[a] < 2 * T;
        key += nk[a][r[a] < 0 ? 0 : (r[a] < T ? 1 : 2)];
    }
    return near ? key : -1;
}

__device__ __forceinline__ void warp_hist_add(int32_t* count, int key) {
    unsigned act = __activemask();
    unsigned peers = __match_any_sync(act, key);
    int lane = threadIdx.x & 31;
    if (lane == __ffs(peers) - 1) atomicAdd(count + key, __popc(peers));
}

// The fields of a simulation and of its species that the particle loop reads,
// staged in shared memory when a CTA's simulation changes, and the unit's
// particle range of each species.  Read from the SimDev in global memory they
// would be fetched again for every particle (the loop's stores to the particle
// arrays might alias them as far as the compiler can tell).
struct HotSp {
    double* src[7];        // read at the particle's place,
    double* dst[7];        // written at its sorted place (the same, unless indirect)
    const int64_t* order;  // where the particle of each sorted place is (nullptr: there)
    const int64_t* id_src;
    int64_t* id_dst;
    int64_t cap;
    int32_t* key;
    int32_t* count;
    const int64_t* off;
    double kq, q;
    int64_t r0, r1;  // the unit's particles
};
struct HotSim {
    double nd[3];
    Amp ja[3];  // current prefactors -1/(dA dt) (2D: jyfac2d for y)
    ExpRange je;
    int T[3], n[3], bsz[3], nb[3], tpb[3], ebs[3];
    int tiles_per_box, ntiles, absorb, ec, jlo, nsp;
    int nk[3][3];  // key parts of the staged tile and its neighbours
    HotSp sp[PIC_MAXSP];
};

// one thread per direction and per species: the loads of different threads overlap
__device__ __forceinline__ void stage_hot(HotSim& h, const SimDev& S) {
    const int a = threadIdx.x, i = (int)threadIdx.x - 4;
    if (a < 3) {
        h.nd[a] = S.nd[a];
        h.T[a] = S.T[a];
        h.n[a] = S.n[a];
        h.bsz[a] = S.bsz[a];
        h.nb[a] = S.nb[a];
        h.tpb[a] = S.tpb[a];
        h.ebs[a] = S.ebs[a];
        h.ja[a] = amp_of(S.dim == 2 && a == 1 ? S.jyfac2d : S.jfac[a]);
    } else if (a == 3) {
        h.tiles_per_box = S.tiles_per_box;
        h.ntiles = S.ntiles;
        h.absorb = S.absorb;
        h.ec = S.ec;
        h.jlo = S.jlo;
        h.nsp = S.nsp;
        h.je = exp_range(S.jfac[0], S.dim == 2 ? S.jyfac2d : S.jfac[1], S.jfac[2]);
    } else if (i < S.nsp) {
        const bool ind = S.sp[i].indirect != 0;
        for (int k = 0; k < 7; ++k) {
            h.sp[i].src[k] = S.sp[i].cur[k];
            h.sp[i].dst[k] = ind ? S.sp[i].alt[k] : S.sp[i].cur[k];
        }
        h.sp[i].order = ind ? S.sp[i].id_alt : nullptr;
        h.sp[i].id_src = S.sp[i].id;
        h.sp[i].cap = S.sp[i].cap;
        h.sp[i].id_dst = S.sp[i].id_alt;
        h.sp[i].key = S.sp[i].key;
        h.sp[i].count = S.sp[i].count;
        h.sp[i].off = S.sp[i].off;
        h.sp[i].kq = S.sp[i].kq;
        h.sp[i].q = S.sp[i].q;
    }
}

// Per-warp buffers of cell-crossing particles in global scratch (struct of
// arrays).  FP64: two stacks in QSLOTS slots, from the bottom the particles that
// cross in one direction, from the top those that cross in several; each is
// drained 32 at a time, and an iteration adds at most 32 in all, so at most
// 31 + 31 + 32 wait.  Linear shapes use the second stack alone: their 54
// contributions on the wide window cost less than the renaming of directions
// (128^3 foil with hot electrons, particle kernel 2.3 against 2.5 ms; cubic
// plasma of 60 x 36 x 50 cells 1.90 with two stacks against 2.16 ms with one).
// FP32: one ring of WQ slots.
constexpr int WQ = 64;
constexpr int QSLOTS = 96;
constexpr int QMAXWARPS = 8;
// queue fields: 0 x^n, 1 z^n, 2 x^{n+1}, 3 z^{n+1} (global, unwrapped), 4 q w,
// 5 y^n (3D) or vy (2D), 6 y^{n+1} (3D)
template <int DIM>
struct QFields {
    static constexpr int n = DIM == 3 ? 7 : 6;
};

static_assert(QFields<3>::n * QSLOTS == PIC_RING_DOUBLES, "a warp's buffer holds 7 fields of QSLOTS slots");

struct SmemPlan {
    int eb_stride;  // doubles per E/B component (multiple of 16 -> 128-byte aligned)
    int eb_vol;
    int pb_off;     // doubles from the base to the particle staging buffers
    int bit_off;    // doubles from the base to the marks of weak cells
    int bit_words;  // words of them per component
    bool staged;    // whether there are such buffers
    size_t bytes;
};

// Particle staging: per warp two buffers of the 7 stored
// values of 32 particles, filled by cp.async one loop iteration ahead.
constexpr int PIN_SLOTS = 7 * 32;
constexpr int PIC_PBUF_DOUBLES = QMAXWARPS * 2 * PIN_SLOTS;

// FP64 converts the staged E/B tile in place to fixed point, the FP32 variant for linear
// shapes to float pairs (F[x], F[x+1] - F[x]), component c at pair c *
// eb_stride, otherwise to floats, component c at float c * eb_stride.
// Layout: E/B tile (TMA) | particle buffers | marks of weak cells.
__host__ __device__ inline SmemPlan smem_plan(const int ebs[3]) {
    SmemPlan p;
    p.eb_vol = ebs[0] * ebs[1] * ebs[2];
    p.eb_stride = (p.eb_vol + 15) & ~15;
    p.pb_off = 6 * p.eb_stride;
    // tiles too large to leave room for the buffers (2D tiles of 64 cells) load
    // their particles directly
    p.bit_words = 2 * ((p.eb_vol + 63) / 64);
    const int bits = 3 * p.bit_words;  // doubles that 6 components' words take
    p.staged = (p.pb_off + PIC_PBUF_DOUBLES + bits) * sizeof(double) <= 225 * 1024;
    p.bit_off = p.pb_off + (p.staged ? PIC_PBUF_DOUBLES : 0);
    p.bytes = (size_t)(p.bit_off + bits) * sizeof(double);
    return p;
}

// double <-> float on the bit patterns without branches: magnitudes below
// 2^-100 (and zero) become a signed zero (an absolute error below 2^-100,
// far inside the FP32 variant's tolerance), larger ones round to 24 bits
__device__ __forceinline__ float f32_of(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned long long u = b & 0x7FFFFFFFFFFFFFFFull;
    const unsigned sgn = (unsigned)(b >> 32) & 0x80000000u;
    const unsigned m = (unsigned)(((u + (1ull << 28)) >> 29) - (896ull << 23));
    return __uint_as_float(sgn | ((u >> 52) >= 1023 - 100 ? m : 0u));
}
__device__ __forceinline__ double f64_of(float f) {
    const unsigned b = __float_as_uint(f), a = b & 0x7FFFFFFFu;
    const unsigned long long sg = (unsigned long long)(b & 0x80000000u) << 32;
    const unsigned long long m = ((unsigned long long)a + (896ull << 23)) << 29;
    return __longlong_as_double((long long)(sg | (a >= 0x00800000u ? m : 0ull)));
}

// Current accumulation.  Every precision adds each contribution to the
// global FP64 J with red.global.add.f64: the add runs in L2, nothing returns
// to the SM, and no FP64 instruction is spent on it.  (A shared-memory FP64
// atomic is a compare-and-swap loop whose retries each cost a full-warp FP64
// add; a shared FP32 atomic add is a compare-and-swap loop as well, measured
// at about 2.3 tries per add on the foil, and moving the FP32 variant's
// current from a shared FP32 tile to these reductions took its particle
// kernel from 895 to 696 us on the 128^3 foil.)  An FP32 value is widened on its bit
// pattern (subnormal floats, below 2^-126, become zero).
__device__ __forceinline__ void red_f64(double* p, double v) {
    asm volatile("red.global.add.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "d"(v) : "memory");
}
__device__ __forceinline__ void jadd(double* p, float v) { red_f64(p, f64_of(v)); }

// Where a tile's current goes: base points at component 0 of local node
// (-jlo, -jlo, -jlo) of the tile (jlo = S.jlo; y is 0 in 2D) in the padded J
// arrays, cs is the component stride, sy and sz the row and plane strides.
// The guard cells (2 to 4 per side) hold the contributions that fall outside
// the domain until the fold kernel adds them to their periodic images.
struct JView {
    double* base;
    int64_t cs;
    int sy, sz;
};

// Esirkepov deposit of one particle into the J arrays (view V) on windows of
// W nodes per direction.  n*: node supports at x^n, m*: at x^{n+1} (local cells).
// Prefix sums of DS along each current's own direction times the transverse
// weight S0a S0b + DSa S0b/2 + S0a DSb/2 + DSa DSb/3 = A_a A_b + DS_a DS_b / 12
// with A = S0 + DS/2.  qw and vy in R; the prefactors -1/(dA dt) come from jf.
template <class R, int DIM, int ORDER, int W, class SV>
__device__ __forceinline__ bool deposit(const SV& S, const JView& V,
                                        R qw, R vy, const R* jf, const Support<ORDER, R>& n0,
                                        const Support<ORDER, R>& n1, const Support<ORDER, R>& n2,
                                        const Support<ORDER, R>& m0, const Support<ORDER, R>& m1,
                                        const Support<ORDER, R>& m2) {
    using A = Arith<R>;
    Window<ORDER, W, R> wx, wy, wz;
    bool ok = make_window<ORDER, W, R>(n0, m0, wx) && make_window<ORDER, W, R>(n2, m2, wz);
    if (DIM == 3) ok = ok && make_window<ORDER, W, R>(n1, m1, wy);
    if (!ok) return false;
    const int sy = V.sy, sz = V.sz, lo = S.jlo;
    double* Jx = V.base;
    double* Jy = V.base + V.cs;
    double* Jz = V.base + 2 * V.cs;
    const R half = A::c(0.5), k12 = A::c(1.0 / 12.0);
    R Ax[W], Az[W], Dx12[W], Dz12[W];
#pragma unroll
    for (int l = 0; l < W; ++l) {
        Ax[l] = fma(half, wx.DS[l], wx.S0[l]);
        Az[l] = fma(half, wz.DS[l], wz.S0[l]);
        Dx12[l] = k12 * wx.DS[l];
        Dz12[l] = k12 * wz.DS[l];
    }
    if constexpr (DIM == 3) {
        R Ay[W];
#pragma unroll
        for (int l = 0; l < W; ++l) Ay[l] = fma(half, wy.DS[l], wy.S0[l]);
        const int bx = wx.base + lo, by = wy.base + lo, bz = wz.base + lo;
        {
            const R c = qw * jf[0];
            R Pf[W - 1];
            R acc = A::c(0.0);
#pragma unroll
            for (int l = 0; l < W - 1; ++l) { acc = acc + wx.DS[l]; Pf[l] = c * acc; }
#pragma unroll
            for (int k = 0; k < W; ++k)
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    const R T = fma(Ay[j], Az[k], wy.DS[j] * Dz12[k]);
                    double* row = Jx + (bz + k) * sz + (by + j) * sy + bx;
#pragma unroll
                    for (int l = 0; l < W - 1; ++l) jadd(row + l, Pf[l] * T);
                }
        }
        {
            const R c = qw * jf[1];
            R Pf[W - 1];
            R acc = A::c(0.0);
#pragma unroll
            for (int j = 0; j < W - 1; ++j) { acc = acc + wy.DS[j]; Pf[j] = c * acc; }
#pragma unroll
            for (int k = 0; k < W; ++k)
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const R T = fma(Ax[i], Az[k], wx.DS[i] * Dz12[k]);
                    double* col = Jy + (bz + k) * sz + by * sy + (bx + i);
#pragma unroll
                    for (int j = 0; j < W - 1; ++j) jadd(col + j * sy, Pf[j] * T);
                }
        }
        {
            const R c = qw * jf[2];
            R Pf[W - 1];
            R acc = A::c(0.0);
#pragma unroll
            for (int k = 0; k < W - 1; ++k) { acc = acc + wz.DS[k]; Pf[k] = c * acc; }
#pragma unroll
            for (int j = 0; j < W; ++j)
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const R T = fma(Ax[i], Ay[j], Dx12[i] * wy.DS[j]);
                    double* col = Jz + bz * sz + (by + j) * sy + (bx + i);
#pragma unroll
                    for (int k = 0; k < W - 1; ++k) jadd(col + k * sz, Pf[k] * T);
                }
        }
    } else {
        const int bx = wx.base + lo, bz = wz.base + lo;
        {  // Jx(i,k) = -(q w /(dz dt)) sum_{i'<=i} DSx(i') (S0z + DSz/2)
            const R c = qw * jf[0];
            R Pf[W - 1];
            R acc = A::c(0.0);
#pragma unroll
            for (int l = 0; l < W - 1; ++l) { acc = acc + wx.DS[l]; Pf[l] = c * acc; }
#pragma unroll
            for (int k = 0; k < W; ++k) {
                double* row = Jx + (bz + k) * sz + bx;
#pragma unroll
                for (int l = 0; l < W - 1; ++l) jadd(row + l, Pf[l] * Az[k]);
            }
        }
        {
            const R c = qw * jf[2];
            R Pf[W - 1];
            R acc = A::c(0.0);
#pragma unroll
            for (int k = 0; k < W - 1; ++k) { acc = acc + wz.DS[k]; Pf[k] = c * acc; }
#pragma unroll
            for (int i = 0; i < W; ++i) {
                double* col = Jz + bz * sz + (bx + i);
#pragma unroll
                for (int k = 0; k < W - 1; ++k) jadd(col + k * sz, Pf[k] * Ax[i]);
            }
        }
        {  // out-of-plane Jy = q w vy / (dx dz) * (Ax Az + DSx DSz / 12)
            const R c = qw * vy * jf[1];
#pragma unroll
            for (int k = 0; k < W; ++k)
#pragma unroll
                for (int i = 0; i < W; ++i)
                    jadd(Jy + (bz + k) * sz + (bx + i), c * fma(Ax[i], Az[k], Dx12[i] * wz.DS[k]));
        }
    }
    return true;
}

// Linear shapes, particle keeping its cell in every direction: the window is
// the two nodes of the cell, DS = (-d, d) with d = f1 - f0, so the prefix sum
// has one term and the transverse weight A_a A_b + DS_a DS_b / 12 is
// A_a A_b +- d_a d_b / 12 (A = (1 - m, m), m = f0 + d/2).  Same weights as
// deposit<R, DIM, 1, 2>, with fewer instructions, given the displacement
// disp[a] = x^{n+1} - x^n (cells) of each direction.
template <class R, int DIM, class SV>
__device__ __forceinline__ void deposit_lin_incell_d(const SV& S, const JView& V,
                                                     R qw, R vy, const R* jf, const Support<1, R>* n,
                                                     const R* disp) {
    using A = Arith<R>;
    const R k12 = A::c(1.0 / 12.0), half = A::c(0.5), one = A::c(1.0);
    const int sy = V.sy, sz = V.sz, lo = S.jlo;
    double* Jx = V.base;
    double* Jy = V.base + V.cs;
    double* Jz = V.base + 2 * V.cs;
    const R dx = disp[0], dz = disp[2];
    const R mx = fma(half, dx, n[0].w[1]), mz = fma(half, dz, n[2].w[1]);
    const R ax0 = one - mx, az0 = one - mz;
    const int bx = n[0].s + lo, bz = n[2].s + lo;
    if constexpr (DIM == 3) {
        // value of node (b, c) of current a: pf_a (A_b A_c + s d_b d_c / 12),
        // s = +1 on the diagonal nodes, -1 off it, pf_a = -q w jf_a d_a; with
        // pe_a = pf_a d_b d_c / 12 = -q w jf_a (d_x d_y d_z / 12) and the node
        // weights (1 - m, m) each value is one FMA of pf_a A_b against A_c
        const R dy = disp[1];
        const R my = fma(half, dy, n[1].w[1]);
        const R ay0 = one - my;
        const int by = n[1].s + lo;
        const R d3 = (dx * dy) * (dz * k12);
        {   // Jx at (bx, by + j, bz + k)
            const R q = qw * jf[0];
            const R pf = -(q * dx), pe = -(q * d3);
            const R p1 = pf * my, p0 = pf - p1;
            double* r = Jx + bz * sz + by * sy + bx;
            jadd(r, fma(p0, az0, pe));
            jadd(r + sy, fma(p1, az0, -pe));
            jadd(r + sz, fma(p0, mz, -pe));
            jadd(r + sz + sy, fma(p1, mz, pe));
        }
        {   // Jy at (bx + i, by, bz + k)
            const R q = qw * jf[1];
            const R pf = -(q * dy), pe = -(q * d3);
            const R p1 = pf * mx, p0 = pf - p1;
            double* r = Jy + bz * sz + by * sy + bx;
            jadd(r, fma(p0, az0, pe));
            jadd(r + 1, fma(p1, az0, -pe));
            jadd(r + sz, fma(p0, mz, -pe));
            jadd(r + sz + 1, fma(p1, mz, pe));
        }
        {   // Jz at (bx + i, by + j, bz)
            const R q = qw * jf[2];
            const R pf = -(q * dz), pe = -(q * d3);
            const R p1 = pf * mx, p0 = pf - p1;
            double* r = Jz + bz * sz + by * sy + bx;
            jadd(r, fma(p0, ay0, pe));
            jadd(r + 1, fma(p1, ay0, -pe));
            jadd(r + sy, fma(p0, my, -pe));
            jadd(r + sy + 1, fma(p1, my, pe));
        }
    } else {
        {   // Jx at (bx, bz + k): -(q w/(dz dt)) DSx A_z
            const R pf = -((qw * jf[0]) * dx);
            double* r = Jx + bz * sz + bx;
            jadd(r, pf * az0);
            jadd(r + sz, pf * mz);
        }
        {   // Jz at (bx + i, bz)
            const R pf = -((qw * jf[2]) * dz);
            double* r = Jz + bz * sz + bx;
            jadd(r, pf * ax0);
            jadd(r + 1, pf * mx);
        }
        {   // out-of-plane Jy at (bx + i, bz + k)
            const R e = (dx * dz) * k12;
            const R c = qw * vy * jf[1];
            double* r = Jy + bz * sz + bx;
            jadd(r, c * fma(ax0, az0, e));
            jadd(r + 1, c * fma(mx, az0, -e));
            jadd(r + sz, c * fma(ax0, mz, -e));
            jadd(r + sz + 1, c * fma(mx, mz, e));
        }
    }
}

// ---- FP64: fixed-point Esirkepov deposit ----------------------------------
// A contribution is amplitude x weight: the weight (the transverse factor, in
// [0, 1]) is a Q62 number, the amplitude (prefactor, q w and the prefix sum of
// DS along the current's direction, or v_y in 2D) an Amp; their product is
// rounded once, to the double that goes to L2.  The weight is good to 8 units of
// 2^-62 (24 for cubic shapes), so a contribution is within 2^-53 of itself and
// 2^-54 of its amplitude, which is what 1 - m alone costs the FP64 factors and
// their four to six roundings.  Nodes that only small weights reach have that
// absolute accuracy, not a relative one.  This takes the deposit off the FP64
// pipe: 36 of about 165 FP64 instructions per particle for linear shapes.
__device__ __forceinline__ void emit(double* p, const Amp& a, q62 T) {
    double v;
    if (contribution(a, T, v)) red_f64(p, v);
}
// amplitudes whose contributions may leave the normal doubles: f, the product
// of the FP64 factors, times the weight
static __device__ __noinline__ void emit_any(double* p, double f, q62 T) {
    red_f64(p, f * ((double)T * 2.168404344971009e-19));  // 2^-62
}

// node shapes of a move on a common window of W nodes: A = (S0 + S1) / 2,
// D = S1 - S0
template <int W>
struct WindowQ {
    int base;
    q62 A[W], D[W];
};
template <int ORDER, int W>
__device__ __forceinline__ bool make_window_q(const SupQ<ORDER>& a, const SupQ<ORDER>& b, WindowQ<W>& win) {
    const int base = min(a.s, b.s);
    const int oa = a.s - base, ob = b.s - base;
    // unsigned: a cell index saturated by a move of 2^31 cells or more wraps the difference
    if ((unsigned)oa > (unsigned)(W - ORDER - 1) || (unsigned)ob > (unsigned)(W - ORDER - 1)) return false;
    win.base = base;
#pragma unroll
    for (int l = 0; l < W; ++l) {
        q62 s0 = 0, s1 = 0;
#pragma unroll
        for (int k = 0; k <= ORDER; ++k) {
            const q62 wa = ORDER == 1 && k == 0 ? kOneQ - a.w[ORDER] : a.w[k];
            const q62 wb = ORDER == 1 && k == 0 ? kOneQ - b.w[ORDER] : b.w[k];
            s0 = (l - oa == k) ? wa : s0;
            s1 = (l - ob == k) ? wb : s1;
        }
        win.A[l] = (s0 + s1) >> 1;
        win.D[l] = s1 - s0;
    }
    return true;
}

// the same for two supports with one first node (W = ORDER + 1)
template <int ORDER>
__device__ __forceinline__ void same_window_q(const SupQ<ORDER>& a, const SupQ<ORDER>& b, WindowQ<ORDER + 1>& win) {
    win.base = a.s;
#pragma unroll
    for (int k = 0; k <= ORDER; ++k) {
        const q62 wa = ORDER == 1 && k == 0 ? kOneQ - a.w[ORDER] : a.w[k];
        const q62 wb = ORDER == 1 && k == 0 ? kOneQ - b.w[ORDER] : b.w[k];
        win.A[k] = (wa + wb) >> 1;
        win.D[k] = wb - wa;
    }
}

constexpr q62 kTwelfthQ = 384307168202282326ll;  // 2^62 / 12

// one current of a deposit: prefix sums of Dp (WP nodes, stride sp) times the
// transverse weight on U x V nodes (strides su, sv)
template <int WP, int WU, int WV>
__device__ __forceinline__ void deposit_current(double* J, const Amp& cw, const q62* Dp, int sp, const WindowQ<WU>& u,
                                                int su, const WindowQ<WV>& v, int sv) {
    Amp pf[WP - 1];
    q62 acc = 0;
#pragma unroll
    for (int l = 0; l < WP - 1; ++l) {
        acc += Dp[l];
        pf[l] = amp_scale(cw, acc);
    }
    Limb Au[WU], Du[WU];
#pragma unroll
    for (int j = 0; j < WU; ++j) {
        Au[j] = limb_of(u.A[j]);
        Du[j] = limb_of(u.D[j]);
    }
    constexpr int UV = WU * WV * (WP - 1) > 12 ? 1 : WV;  // long windows: a loop
#pragma unroll UV
    for (int k = 0; k < WV; ++k) {
        q62 va = v.A[0], vd = v.D[0];
#pragma unroll
        for (int i = 1; i < WV; ++i) {
            va = k == i ? v.A[i] : va;
            vd = k == i ? v.D[i] : vd;
        }
        const Limb ak = limb_of(va), dk = limb_of(mulq(limb_of(vd), limb_of(kTwelfthQ)));
#pragma unroll
        for (int j = 0; j < WU; ++j) {
            AccQ s;
            s.mac(Au[j], ak);
            s.mac(Du[j], dk);
            double* row = J + k * sv + j * su;
#pragma unroll
            for (int l = 0; l < WP - 1; ++l) emit(row + l * sp, pf[l], s.get());
        }
    }
}

// Deposit of a particle that changes its support along one direction, a: only
// that direction needs the ORDER + 2 window.  The directions are renamed per
// particle (a, and the transverse b < c), so that one code serves all three:
// 20 contributions for linear shapes against 54 on three ORDER + 2 windows (75
// against 144 quadratic, 184 against 300 cubic).
template <int DIM, int ORDER>
__device__ __forceinline__ void deposit_one_axis(int lo, const JView& V, const Amp* ja, double qw, double vy,
                                                 const SupQ<ORDER>* n, const SupQ<ORDER>* m, int a) {
    constexpr int WA = ORDER + 2, WB = ORDER + 1;
    const int b = DIM == 2 ? 2 - a : (a == 0 ? 1 : 0), c = a == 2 ? 1 : 2;
    const Amp q = amp_of(qw);
    double* J0 = V.base + (min(n[2].s, m[2].s) + lo) * V.sz + (min(n[0].s, m[0].s) + lo);
    if (DIM == 3) J0 += (min(n[1].s, m[1].s) + lo) * V.sy;
    const int sa = pick3(a, 1, V.sy, V.sz), sb = pick3(b, 1, V.sy, V.sz), sc = pick3(c, 1, V.sy, V.sz);
    WindowQ<WA> wa;
    WindowQ<WB> wb, wc;
    if constexpr (DIM == 3) {
        make_window_q<ORDER, WA>(pick3(a, n[0], n[1], n[2]), pick3(a, m[0], m[1], m[2]), wa);
        same_window_q<ORDER>(b == 0 ? n[0] : n[1], b == 0 ? m[0] : m[1], wb);
        same_window_q<ORDER>(c == 1 ? n[1] : n[2], c == 1 ? m[1] : m[2], wc);
        deposit_current<WA, WB, WB>(J0 + a * V.cs, amp_mul(pick3(a, ja[0], ja[1], ja[2]), q), wa.D, sa, wb, sb, wc, sc);
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {  // the currents along b and along c
            const int d = i == 0 ? b : c;
            WindowQ<WB> p = wb, t = wc;
            if (i != 0) {
                p = wc;
                t = wb;
            }
            deposit_current<WB, WB, WA>(J0 + d * V.cs, amp_mul(pick3(d, ja[0], ja[1], ja[2]), q), p.D,
                                        i == 0 ? sb : sc, t, i == 0 ? sc : sb, wa, sa);
        }
    } else {
        make_window_q<ORDER, WA>(a == 0 ? n[0] : n[2], a == 0 ? m[0] : m[2], wa);
        same_window_q<ORDER>(a == 0 ? n[2] : n[0], a == 0 ? m[2] : m[0], wb);
        const Amp ca = amp_mul(a == 0 ? ja[0] : ja[2], q), cb = amp_mul(a == 0 ? ja[2] : ja[0], q);
        double* Ja = J0 + a * V.cs;
        double* Jb = J0 + b * V.cs;
        q62 acc = 0;
#pragma unroll
        for (int l = 0; l < WA - 1; ++l) {
            acc += wa.D[l];
            const Amp pf = amp_scale(ca, acc);
#pragma unroll
            for (int j = 0; j < WB; ++j) emit(Ja + l * sa + j * sb, pf, wb.A[j]);
        }
        acc = 0;
#pragma unroll
        for (int l = 0; l < WB - 1; ++l) {
            acc += wb.D[l];
            const Amp pf = amp_scale(cb, acc);
#pragma unroll
            for (int j = 0; j < WA; ++j) emit(Jb + l * sb + j * sa, pf, wa.A[j]);
        }
        const Amp cv = amp_mul(amp_mul(ja[1], q), amp_of(vy));
#pragma unroll 1
        for (int k = 0; k < WB; ++k) {
            q62 va = wb.A[0], vd = wb.D[0];
#pragma unroll
            for (int i = 1; i < WB; ++i) {
                va = k == i ? wb.A[i] : va;
                vd = k == i ? wb.D[i] : vd;
            }
            const Limb ak = limb_of(va), dk = limb_of(mulq(limb_of(vd), limb_of(kTwelfthQ)));
#pragma unroll
            for (int i = 0; i < WA; ++i) {
                AccQ s;
                s.mac(limb_of(wa.A[i]), ak);
                s.mac(limb_of(wa.D[i]), dk);
                emit(J0 + V.cs + k * sb + i * sa, cv, s.get());
            }
        }
    }
}

// Deposit on windows of W nodes per direction: for each current (a loop: one
// copy of the code, whose size the instruction cache feels) the prefix sums of
// D along its own direction times the transverse weight A_b A_c + D_b D_c / 12.
// ANY: amplitudes of any size (emit_any).
template <int DIM, int ORDER, int W, bool ANY>
__device__ __forceinline__ bool deposit_q(int lo, const JView& V, const Amp* ja, const double* jf, double qw,
                                          double vy, const SupQ<ORDER>* n, const SupQ<ORDER>* m) {
    WindowQ<W> w0, w1, w2;
    if constexpr (W == ORDER + 1) {  // the support stays
        same_window_q<ORDER>(n[0], m[0], w0);
        same_window_q<ORDER>(n[2], m[2], w2);
        if (DIM == 3) same_window_q<ORDER>(n[1], m[1], w1);
    } else {
        bool ok = make_window_q<ORDER, W>(n[0], m[0], w0) && make_window_q<ORDER, W>(n[2], m[2], w2);
        if (DIM == 3) ok = ok && make_window_q<ORDER, W>(n[1], m[1], w1);
        if (!ok) return false;
    }
    constexpr int UW = ANY ? 1 : W;                     // inner loops: unrolled, but for the rare case
    constexpr int UK = ANY || ORDER > 1 ? 1 : W;        // outer transverse loop: rolled for long windows
    double* origin = V.base + (w2.base + lo) * V.sz + (w0.base + lo);
    if (DIM == 3) origin += (w1.base + lo) * V.sy;
    const Amp q = amp_of(qw);
    auto out = [&](double* p, const Amp& a, q62 T, double f) {
        if constexpr (ANY) emit_any(p, f, max(T, 0ll));
        else emit(p, a, T);
    };
    if constexpr (DIM == 3) {
#pragma unroll 1
        for (int a = 0; a < 3; ++a) {
            const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
            const int sa = pick3(a, 1, V.sy, V.sz), sb = pick3(b, 1, V.sy, V.sz), sc = pick3(c, 1, V.sy, V.sz);
            const Amp cw = amp_mul(pick3(a, ja[0], ja[1], ja[2]), q);
            const double cf = ANY ? pick3(a, jf[0], jf[1], jf[2]) * qw : 0.0;
            Amp pf[W - 1];
            double nf[W - 1];
            Limb Ab[W], Db[W], Ac[W], Dc[W];
            q62 acc = 0;
#pragma unroll
            for (int l = 0; l < W; ++l) {
                if (l < W - 1) {
                    acc += pick3(a, w0.D[l], w1.D[l], w2.D[l]);
                    pf[l] = amp_scale(cw, acc);
                    nf[l] = ANY ? cf * ((double)acc * 2.168404344971009e-19) : 0.0;
                }
                Ab[l] = limb_of(b == 0 ? w0.A[l] : w1.A[l]);
                Db[l] = limb_of(b == 0 ? w0.D[l] : w1.D[l]);
                Ac[l] = limb_of(c == 1 ? w1.A[l] : w2.A[l]);
                Dc[l] = limb_of(mulq(limb_of(c == 1 ? w1.D[l] : w2.D[l]), limb_of(kTwelfthQ)));
            }
            double* Ja = origin + a * V.cs;
#pragma unroll UK
            for (int k = 0; k < W; ++k) {
                Limb ak = Ac[0], dk = Dc[0];
#pragma unroll
                for (int i = 1; i < W; ++i) {
                    ak = k == i ? Ac[i] : ak;
                    dk = k == i ? Dc[i] : dk;
                }
                double* plane = Ja + k * sc;
#pragma unroll UW
                for (int j = 0; j < W; ++j) {
                    AccQ s;
                    s.mac(Ab[j], ak);
                    s.mac(Db[j], dk);
                    const q62 T = s.get();
                    double* row = plane + j * sb;
#pragma unroll UW
                    for (int l = 0; l < W - 1; ++l) out(row + l * sa, pf[l], T, nf[l]);
                }
            }
        }
    } else {
#pragma unroll 1
        for (int a = 0; a < 2; ++a) {  // Jx, then Jz: the transverse weight is A
            const int sa = a == 0 ? 1 : V.sz, sb = a == 0 ? V.sz : 1;
            const Amp cw = amp_mul(a == 0 ? ja[0] : ja[2], q);
            const double cf = ANY ? (a == 0 ? jf[0] : jf[2]) * qw : 0.0;
            double* Ja = origin + (a == 0 ? 0 : 2 * V.cs);
            q62 acc = 0;
#pragma unroll UW
            for (int l = 0; l < W - 1; ++l) {
                acc += a == 0 ? w0.D[l] : w2.D[l];
                const Amp pf = amp_scale(cw, acc);
                const double nf = ANY ? cf * ((double)acc * 2.168404344971009e-19) : 0.0;
#pragma unroll UW
                for (int j = 0; j < W; ++j) out(Ja + j * sb + l * sa, pf, a == 0 ? w2.A[j] : w0.A[j], nf);
            }
        }
        // out-of-plane Jy = q w vy / (dx dz) (Ax Az + Dx Dz / 12)
        const Amp cv = amp_mul(amp_mul(ja[1], q), amp_of(vy));
        const double nfy = ANY ? jf[1] * qw * vy : 0.0;
        double* Jy = origin + V.cs;
#pragma unroll UW
        for (int k = 0; k < W; ++k) {
            const Limb ak = limb_of(w2.A[k]), dk = limb_of(mulq(limb_of(w2.D[k]), limb_of(kTwelfthQ)));
#pragma unroll UW
            for (int i = 0; i < W; ++i) {
                AccQ s;
                s.mac(limb_of(w0.A[i]), ak);
                s.mac(limb_of(w0.D[i]), dk);
                out(Jy + k * V.sz + i, cv, s.get(), nfy);
            }
        }
    }
    return true;
}

// whether every amplitude of a particle stays inside the normal doubles (a zero
// q w or v_y deposits nothing, and is)
template <int DIM>
__device__ __forceinline__ bool amps_safe(const ExpRange& r, double qw, double vy) {
    const int eq = exp_field(qw);
    bool ok = in_range(r, eq);
    if (DIM == 2) {
        const int ev = exp_field(vy);
        ok = ok && (vy == 0.0 || (ev > 0 && ev < 0x7FF && in_range(r, eq + ev - 1023)));
    }
    return ok || qw == 0.0;
}

// Linear shapes, particle keeping its cell: the window is the two nodes of the
// cell, D = (-d, d), one prefix sum, and with the mid-path offsets m and
// P = m_b m_c + d_b d_c / 12 the four weights are P, m_b - P, m_c - P and
// 1 - m_b - m_c + P (exactly zero where they should be: a particle on a node and
// moving along no other direction gives its other nodes nothing).  cw: prefactor x
// q w per current (2D: x v_y for y).
template <int DIM>
__device__ __forceinline__ void deposit_lin_q(int lo, const JView& V, const Amp* cw, const SupQ<1>* n,
                                              const SupQ<1>* mv) {
    q62 d[3], m[3];
    Limb lm[3], l12[3], ld[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) continue;
        d[a] = mv[a].w[1] - n[a].w[1];
        m[a] = (n[a].w[1] + mv[a].w[1]) >> 1;
        lm[a] = limb_of(m[a]);
        ld[a] = limb_of(d[a]);
        if (a > 0) l12[a] = limb_of(mulq(ld[a], limb_of(kTwelfthQ)));
    }
    double* origin = V.base + (n[2].s + lo) * V.sz + (n[0].s + lo);
    if (DIM == 3) origin += (n[1].s + lo) * V.sy;
    auto four = [&](double* r, const Amp& pf, q62 mb, q62 mc, const Limb& lb, const Limb& lc, const Limb& db,
                    const Limb& dc12, int sb, int sc) {
        AccQ s;
        s.mac(lb, lc);
        s.mac(db, dc12);
        const q62 P = s.get();
        emit(r, pf, kOneQ - mb - mc + P);
        emit(r + sb, pf, mb - P);
        emit(r + sc, pf, mc - P);
        emit(r + sb + sc, pf, P);
    };
    if constexpr (DIM == 3) {
        // a loop: the instruction cache feels three copies (128^3 foil 1567 -> 1524 us)
#pragma unroll 1
        for (int a = 0; a < 3; ++a) {
            const Amp pf = amp_scale(pick3(a, cw[0], cw[1], cw[2]), -pick3(a, d[0], d[1], d[2]));
            four(origin + a * V.cs, pf, a == 0 ? m[1] : m[0], a == 2 ? m[1] : m[2], a == 0 ? lm[1] : lm[0],
                 a == 2 ? lm[1] : lm[2], a == 0 ? ld[1] : ld[0], a == 2 ? l12[1] : l12[2], a == 0 ? V.sy : 1,
                 a == 2 ? V.sy : V.sz);
        }
    } else {
        const Amp px = amp_scale(cw[0], -d[0]), pz = amp_scale(cw[2], -d[2]);
        emit(origin, px, kOneQ - m[2]);
        emit(origin + V.sz, px, m[2]);
        emit(origin + 2 * V.cs, pz, kOneQ - m[0]);
        emit(origin + 2 * V.cs + 1, pz, m[0]);
        four(origin + V.cs, cw[1], m[0], m[2], lm[0], lm[2], ld[0], l12[2], 1, V.sz);
    }
}

// node supports of a move, from the positions
template <int DIM, int ORDER>
__device__ __forceinline__ void node_supports_q(const double* x, const int* o, SupQ<ORDER>* n, bool& nan) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) continue;
        const CellQ c = cell_q(x[a]);
        nan = nan || c.nan;
        n[a] = node_support<ORDER>(c, o[a]);
    }
}

// any particle's deposit on the ORDER + 2 window with amplitudes of any size
// (weights or prefactors near the ends of the double range, Inf, NaN)
template <int DIM, int ORDER>
static __device__ __noinline__ bool deposit_any(const SimDev& S, JView V, int ox, int oy, int oz, double X, double Y,
                                                double Z, double X1, double Y1, double Z1, double qw, double vy) {
    const int o[3] = {ox, oy, oz};
    const double x0[3] = {X, Y, Z}, x1[3] = {X1, Y1, Z1};
    const double jf[3] = {S.jfac[0], DIM == 3 ? S.jfac[1] : S.jyfac2d, S.jfac[2]};
    const Amp ja[3] = {amp_of(jf[0]), amp_of(jf[1]), amp_of(jf[2])};
    SupQ<ORDER> n[3], m[3];
    bool nan = false;
    node_supports_q<DIM, ORDER>(x0, o, n, nan);
    node_supports_q<DIM, ORDER>(x1, o, m, nan);
    return deposit_q<DIM, ORDER, ORDER + 2, true>(S.jlo, V, ja, jf, nan ? qw * __longlong_as_double(0x7FF8000000000000ll) : qw,
                                                  vy, n, m);
}

// One particle's stored state as read from HBM (positions in global cell
// units, momenta and weight as stored); loaded ahead of its push so that the
// loads of several particles per thread can be in flight together.
struct PIn {
    double X, Y, Z, u0, u1, u2, w;
};

template <int DIM, class SPV>
__device__ __forceinline__ PIn load_one(const SPV& sp, int64_t p) {
    PIn in;
    in.X = sp.src[0][p];
    in.Y = (DIM == 3) ? sp.src[1][p] : 0.0;
    in.Z = sp.src[2][p];
    in.u0 = sp.src[3][p];
    in.u1 = sp.src[4][p];
    in.u2 = sp.src[5][p];
    in.w = sp.src[6][p];
    return in;
}

// The same values staged through shared memory: the lane's column of a
// staging buffer (value a of the particle at slot[32 a]), filled by cp.async
template <int DIM, class SPV>
__device__ __forceinline__ void stage_in(const SPV& sp, int64_t p, double* slot) {
#pragma unroll
    for (int a = 0; a < 7; ++a)
        if (DIM == 3 || a != 1) cp_async_8(slot + 32 * a, sp.src[a] + p);
}
template <int DIM>
__device__ __forceinline__ PIn read_staged(const double* slot) {
    PIn in;
    in.X = slot[0];
    in.Y = (DIM == 3) ? slot[32] : 0.0;
    in.Z = slot[64];
    in.u0 = slot[96];
    in.u1 = slot[128];
    in.u2 = slot[160];
    in.w = slot[192];
    return in;
}

// Gather, Boris push, and deposit of one particle, FP64.  The gather and the
// deposit are fixed-point; emax: biased exponents of the staged tile's components;
// weak: marks where a component is gathered by itself, nullptr if there is none.
template <class R, int DIM, int ORDER, class SV, class SPV>
__device__ __forceinline__ void push_one_q(const SV& S, const SPV& sp, const SimDev& SG, const Tile& tl,
                                           const double* __restrict__ sEB, const unsigned* __restrict__ weak,
                                           const int* __restrict__ emax,
                                           const JView& V, double* __restrict__ sQw, unsigned* s_one, unsigned* s_many,
                                           const SmemPlan& P, const R* dtd, R kq, double qs, int64_t p, const PIn& in,
                                           int32_t* err) {
    using A = Arith<R>;
    const double x0[3] = {in.X, DIM == 3 ? in.Y : 0.0, in.Z};
    double qw = qs * in.w;

    // ---- gather at x^n: node and half-node supports per direction (tile-local nodes)
    SupQ<ORDER> nd[3];
    Six f;
    {
        AxisQ<ORDER> na[3], ha[3];
        bool inside = true, nan = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (DIM == 2 && a == 1) continue;
            const CellQ c = cell_q(x0[a]);
            nan = nan || c.nan;
            inside = inside && (unsigned)(c.i - tl.o[a]) < (unsigned)S.T[a];
            nd[a] = node_support<ORDER>(c, tl.o[a]);
            na[a] = axis_of<ORDER>(nd[a]);
            ha[a] = axis_of<ORDER>(half_support<ORDER>(c, tl.o[a], S.ec != 0));
        }
        if (!inside) {
            // the particle must sit in its tile; the E/B halo then covers every support above
            atomicOr(err, PIC_DERR_BOUNDS);
            sp.key[p] = S.ntiles;
            warp_hist_add(sp.count, S.ntiles);
            return;
        }
        f = gather6_q<ORDER, DIM>(reinterpret_cast<const long long*>(sEB), P.eb_stride, S.ebs[0], S.ebs[1], emax, na, ha);
        if (weak) {
            unsigned mask = weak_components<ORDER, DIM>(weak, P.bit_words, S.ebs[0], S.ebs[1], nd, ha);
            while (mask != 0u) {
                const int c = __ffs((int)mask) - 1;
                mask &= mask - 1u;
                const double v = gather1_weak<ORDER, DIM>(SG, c, x0[0], x0[1], x0[2], tl.o[0], tl.o[1], tl.o[2]);
#pragma unroll
                for (int k = 0; k < 6; ++k) f.v[k] = c == k ? v : f.v[k];
            }
        }
        if (nan) f.v[0] = f.v[1] = f.v[2] = __longlong_as_double(0x7FF8000000000000ll);
    }
    const R u0 = A::from(in.u0), u1 = A::from(in.u1), u2 = A::from(in.u2);
    const R e0 = A::from(f.v[0]), e1 = A::from(f.v[1]), e2 = A::from(f.v[2]);
    const R b0 = A::from(f.v[3]), b1 = A::from(f.v[4]), b2 = A::from(f.v[5]);

    // ---- relativistic Boris push
    const R one = A::c(1.0);
    const R m0 = fma(kq, e0, u0), m1 = fma(kq, e1, u1), m2 = fma(kq, e2, u2);
    const R ig = A::rsqrt(fma(m2, m2, fma(m1, m1, fma(m0, m0, one))));
    const R kg = kq * ig;
    const R t0 = kg * b0, t1 = kg * b1, t2 = kg * b2;
    const R sf = A::two_over(fma(t2, t2, fma(t1, t1, fma(t0, t0, one))));
    const R s0 = sf * t0, s1 = sf * t1, s2 = sf * t2;
    // u' = u- + u- x t, u+ = u- + u' x s, each component as two FMAs
    const R d0 = fma(m1, t2, fma(-m2, t1, m0));
    const R d1 = fma(m2, t0, fma(-m0, t2, m1));
    const R d2 = fma(m0, t1, fma(-m1, t0, m2));
    const R p0 = fma(d1, s2, fma(-d2, s1, m0));
    const R p1 = fma(d2, s0, fma(-d0, s2, m1));
    const R p2 = fma(d0, s1, fma(-d1, s0, m2));
    const R n0 = fma(kq, e0, p0), n1 = fma(kq, e1, p1), n2 = fma(kq, e2, p2);
    const R ign = A::rsqrt(fma(n2, n2, fma(n1, n1, fma(n0, n0, one))));
    const R v1 = n1 * ign;
    double x1[3];
    x1[0] = A::move(n0 * ign, dtd[0], x0[0]);
    x1[1] = DIM == 3 ? A::move(v1, dtd[1], x0[1]) : 0.0;
    x1[2] = A::move(n2 * ign, dtd[2], x0[2]);
    const double vy = DIM == 3 ? 0.0 : A::to(v1);

    // ---- Esirkepov deposit of J^{n+1/2} from x^n to x^{n+1}
    SupQ<ORDER> mv[3];
    int g[3] = {0, 0, 0};
    int ncross = 0;  // directions in which the support moves
    bool nan = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) continue;
        const CellQ c = cell_q(x1[a]);
        nan = nan || c.nan;
        g[a] = c.i;
        mv[a] = node_support<ORDER>(c, tl.o[a]);
        ncross += mv[a].s == nd[a].s ? 0 : 1;
    }
    if (nan) qw = __longlong_as_double(0x7FF8000000000000ll);
    if (ncross == 0) {
        const bool ok = amps_safe<DIM>(S.je, qw, vy);
        if constexpr (ORDER == 1) {
            if (ok) {
                const Amp q = amp_of(qw);
                Amp cw[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) cw[a] = amp_mul(S.ja[a], q);
                if (DIM == 2) cw[1] = amp_mul(cw[1], amp_of(vy));
                deposit_lin_q<DIM>(S.jlo, V, cw, nd, mv);
            }
        } else {
            if (ok) deposit_q<DIM, ORDER, ORDER + 1, false>(S.jlo, V, S.ja, nullptr, qw, vy, nd, mv);
        }
        if (!ok)
            deposit_any<DIM, ORDER>(SG, V, tl.o[0], tl.o[1], tl.o[2], x0[0], x0[1], x0[2], x1[0], x1[1], x1[2], qw, vy);
    } else {
        const int slot = ORDER > 1 && ncross == 1 ? (int)atomicAdd(s_one, 1u) : QSLOTS - 1 - (int)atomicAdd(s_many, 1u);
        sQw[0 * QSLOTS + slot] = x0[0];
        sQw[1 * QSLOTS + slot] = x0[2];
        sQw[2 * QSLOTS + slot] = x1[0];
        sQw[3 * QSLOTS + slot] = x1[2];
        sQw[4 * QSLOTS + slot] = qw;
        sQw[5 * QSLOTS + slot] = DIM == 3 ? x0[1] : vy;
        if (DIM == 3) sQw[6 * QSLOTS + slot] = x1[1];
    }

    // ---- new position, boundary, re-sort key
    auto wrap = [&](int a) {
        if (is_neg(x1[a]) || ge_pos(x1[a], S.nd[a])) x1[a] = wrap_periodic(x1[a], S.nd[a]);
    };
    const int r[3] = {g[0] - tl.o[0], g[1] - tl.o[1], g[2] - tl.o[2]};
    int key = near_key<DIM>(S, S.nk, r);
    // z < A or z >= n - A for integer bounds: compare floor(z)
    if (S.absorb > 0 && (g[2] < S.absorb || g[2] >= S.n[2] - S.absorb)) key = S.ntiles;
    wrap(0);
    if (DIM == 3) wrap(1);
    if (S.absorb <= 0) wrap(2);
    if (key < 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) g[a] = DIM == 3 || a != 1 ? min(max(ifloor(x1[a]), 0), S.n[a] - 1) : 0;
        key = tile_key(S, g[0], g[1], g[2]);
    }
    sp.dst[0][p] = x1[0];
    if (DIM == 3) sp.dst[1][p] = x1[1];
    sp.dst[2][p] = x1[2];
    sp.dst[3][p] = A::to(n0);
    sp.dst[4][p] = A::to(n1);
    sp.dst[5][p] = A::to(n2);
    sp.key[p] = key;
    warp_hist_add(sp.count, key);
}

// The same in FP32 (R = float), quadratic and cubic shapes.  Particles that keep their
// support in every direction deposit at once on the small window; the others
// go to the warp's ring buffer, drained 32 at a time by drain_warp.
template <class R, int DIM, int ORDER, class SV, class SPV>
__device__ __forceinline__ void push_one(const SV& S, const SPV& sp, const Tile& tl,
                                         const R* __restrict__ sEB, const JView& V,
                                         double* __restrict__ sQw, unsigned* s_tail, const SmemPlan& P,
                                         const R* jf, const R* dtd, R kq, R qs, int64_t p, const PIn& in,
                                         int32_t* err) {
    using A = Arith<R>;
    double X = in.X, Z = in.Z;
    double Y = (DIM == 3) ? in.Y : 0.0;
    const R u0 = A::from(in.u0), u1 = A::from(in.u1), u2 = A::from(in.u2);
    const R qw = qs * A::from(in.w);

    // ---- gather at x^n: node and half-node supports per direction (tile-local nodes)
    Support<ORDER, R> nd[3], hf[3];
    int cx, cy = 0, cz;
    const bool ec = S.ec != 0;
    supports_at<ORDER, R>(X, tl.o[0], ec, nd[0], hf[0], cx);
    supports_at<ORDER, R>(Z, tl.o[2], ec, nd[2], hf[2], cz);
    if (DIM == 3) {
        supports_at<ORDER, R>(Y, tl.o[1], ec, nd[1], hf[1], cy);
    } else {
        nd[1].s = -1;
        nd[1].w[0] = A::c(1.0);
        hf[1] = nd[1];
    }
    {
        // the particle must sit in its tile (local cell index in [0, T)); the
        // E/B halo then covers every support above
        bool in = cx >= 0 && cx < S.T[0] && cz >= 0 && cz < S.T[2];
        if (DIM == 3) in = in && cy >= 0 && cy < S.T[1];
        if (!in) {
            atomicOr(err, PIC_DERR_BOUNDS);
            sp.key[p] = S.ntiles;
            warp_hist_add(sp.count, S.ntiles);
            return;
        }
    }
    const int SX = S.ebs[0], SY = S.ebs[1];
    R ev[3], bv[3];
    gather6<R, ORDER, DIM>(sEB, P.eb_stride, SX, SY, nd, hf, ev, bv);
    const R e0 = ev[0], e1 = ev[1], e2 = ev[2], b0 = bv[0], b1 = bv[1], b2 = bv[2];

    // ---- relativistic Boris push
    const R one = A::c(1.0);
    const R m0 = fma(kq, e0, u0), m1 = fma(kq, e1, u1), m2 = fma(kq, e2, u2);
    const R ig = A::rsqrt(fma(m2, m2, fma(m1, m1, fma(m0, m0, one))));
    const R kg = kq * ig;
    const R t0 = kg * b0, t1 = kg * b1, t2 = kg * b2;
    const R t2n = fma(t2, t2, fma(t1, t1, t0 * t0));
    const R sf = A::two_over(one + t2n);
    const R s0 = sf * t0, s1 = sf * t1, s2 = sf * t2;
    // u' = u- + u- x t, u+ = u- + u' x s, each component as two FMAs
    const R d0 = fma(m1, t2, fma(-m2, t1, m0));
    const R d1 = fma(m2, t0, fma(-m0, t2, m1));
    const R d2 = fma(m0, t1, fma(-m1, t0, m2));
    const R p0 = fma(d1, s2, fma(-d2, s1, m0));
    const R p1 = fma(d2, s0, fma(-d0, s2, m1));
    const R p2 = fma(d0, s1, fma(-d1, s0, m2));
    const R n0 = fma(kq, e0, p0), n1 = fma(kq, e1, p1), n2 = fma(kq, e2, p2);
    const R ign = A::rsqrt(fma(n2, n2, fma(n1, n1, fma(n0, n0, one))));
    const R v1 = n1 * ign;
    const double dX = A::to((n0 * ign) * dtd[0]), dZ = A::to((n2 * ign) * dtd[2]);
    const double dY = (DIM == 3) ? A::to(v1 * dtd[1]) : 0.0;

    // ---- Esirkepov deposit of J^{n+1/2} from x^n to x^{n+1}
    const double X1 = X + dX, Z1 = Z + dZ;
    const double Y1 = (DIM == 3) ? Y + dY : 0.0;
    Support<ORDER, R> mv[3];
    mv[0] = support_at<ORDER, R>(X1, tl.o[0]);
    mv[2] = support_at<ORDER, R>(Z1, tl.o[2]);
    if (DIM == 3) mv[1] = support_at<ORDER, R>(Y1, tl.o[1]);
    else mv[1] = nd[1];
    bool same = mv[0].s == nd[0].s && mv[2].s == nd[2].s && (DIM == 2 || mv[1].s == nd[1].s);
    if (same) {
        deposit<R, DIM, ORDER, ORDER + 1>(S, V, qw, v1, jf, nd[0], nd[1], nd[2], mv[0], mv[1], mv[2]);
    } else {
        // the ring never holds more than 31 + 32 entries: the warp drains 32
        // whenever 32 are waiting
        const unsigned slot = atomicAdd(s_tail, 1u) & (WQ - 1);
        sQw[0 * WQ + slot] = X;
        sQw[1 * WQ + slot] = Z;
        sQw[2 * WQ + slot] = X1;
        sQw[3 * WQ + slot] = Z1;
        sQw[4 * WQ + slot] = A::to(qw);
        sQw[5 * WQ + slot] = DIM == 3 ? Y : A::to(v1);
        if (DIM == 3) sQw[6 * WQ + slot] = Y1;
    }

    // ---- new position, boundary, re-sort key
    X = X1;
    Z = Z1;
    if (is_neg(X) || ge_pos(X, S.nd[0])) X = wrap_periodic(X, S.nd[0]);
    if (DIM == 3) {
        Y = Y1;
        if (is_neg(Y) || ge_pos(Y, S.nd[1])) Y = wrap_periodic(Y, S.nd[1]);
    }
    int key = -1;
    if (S.absorb > 0) {
        // z < A or z >= n - A for integer bounds: compare floor(z)
        const int iz = ifloor(Z);
        if (iz < S.absorb || iz >= S.n[2] - S.absorb) key = S.ntiles;
    } else {
        if (is_neg(Z) || ge_pos(Z, S.nd[2])) Z = wrap_periodic(Z, S.nd[2]);
    }
    if (key < 0) {
        int ix = min(max(ifloor(X), 0), S.n[0] - 1);
        int iy = (DIM == 3) ? min(max(ifloor(Y), 0), S.n[1] - 1) : 0;
        int iz = min(max(ifloor(Z), 0), S.n[2] - 1);
        // most particles stay in their tile: its key without the divisions
        bool own = (unsigned)(ix - tl.o[0]) < (unsigned)S.T[0] && (unsigned)(iz - tl.o[2]) < (unsigned)S.T[2];
        if (DIM == 3) own = own && (unsigned)(iy - tl.o[1]) < (unsigned)S.T[1];
        key = own ? tl.t : tile_key(S, ix, iy, iz);
    }
    sp.dst[0][p] = X;
    if (DIM == 3) sp.dst[1][p] = Y;
    sp.dst[2][p] = Z;
    sp.dst[3][p] = A::to(n0);
    sp.dst[4][p] = A::to(n1);
    sp.dst[5][p] = A::to(n2);
    sp.key[p] = key;
    warp_hist_add(sp.count, key);
}

// ---- FP32 variant, linear shapes: positions in 24-bit fixed point --------
// Adding M = 1.5 * 2^28 to a position X (cells, |X| < 2^27), rounded toward
// -infinity, truncates it to a multiple of 2^-24 and leaves it, as a
// fixed-point number with 24 fractional bits, in the low bits of the sum: one
// FP64 add gives the cell (the bits above 24: floor(X) exactly, negative X
// too) and the in-cell offset (the low 24) with integer instructions and no
// branches.  The move is carried in the same units (d rounded to 2^-24 of a
// cell), so the cell test of x^{n+1}, the in-cell displacement used by the
// deposit and the stored FP64 position agree exactly; after the first step
// every stored position lies on the 2^-24 grid.
constexpr double kFixM = 402653184.0;  // 1.5 * 2^28: ulp 2^-24 over [2^28, 2^29)
__device__ __forceinline__ long long fix24(double x) {
    return __double_as_longlong(__dadd_rd(x, kFixM)) - __double_as_longlong(kFixM);
}
__device__ __forceinline__ double unfix24(long long b) {
    return __longlong_as_double(b + __double_as_longlong(kFixM)) - kFixM;  // exact
}
__device__ __forceinline__ float frac24(long long b) { return (float)(int)(b & 0xFFFFFFll) * 5.9604644775390625e-8f; }

// Linear FP32 gather from the staged tile held as pairs (F[x], F[x+1] - F[x])
// of floats: each x lerp is one 8-byte shared load and one FMA, and gives the
// same float as a + f (b - a) on the two floats.  Component c starts at pair
// c * stride.
template <int DIM>
__device__ __forceinline__ float interp_pairs(const float2* __restrict__ F, int SX, int SY, const Support<1, float>& sx,
                                              const Support<1, float>& sy, const Support<1, float>& sz) {
    constexpr int H = EBHalo<1>::lo;
    auto lerp = [](float a, float b, float f) { return fmaf(f, b - a, a); };
    const float fx = sx.w[1];
    if constexpr (DIM == 3) {
        const float2* r = F + ((sz.s + H) * SY + (sy.s + H)) * SX + (sx.s + H);
        const float2 p00 = r[0], p10 = r[SX], p01 = r[SX * SY], p11 = r[SX * SY + SX];
        const float a00 = fmaf(fx, p00.y, p00.x), a10 = fmaf(fx, p10.y, p10.x);
        const float a01 = fmaf(fx, p01.y, p01.x), a11 = fmaf(fx, p11.y, p11.x);
        return lerp(lerp(a00, a10, sy.w[1]), lerp(a01, a11, sy.w[1]), sz.w[1]);
    } else {
        const float2* r = F + (sz.s + H) * SX + (sx.s + H);
        const float2 p0 = r[0], p1 = r[SX];
        return lerp(fmaf(fx, p0.y, p0.x), fmaf(fx, p1.y, p1.x), sz.w[1]);
    }
}
template <int DIM>
__device__ __forceinline__ void gather6_pairs(const float2* __restrict__ sP, int stride, int SX, int SY,
                                              const Support<1, float>* nd, const Support<1, float>* hf, float* e,
                                              float* b) {
    e[0] = interp_pairs<DIM>(sP, SX, SY, hf[0], nd[1], nd[2]);
    e[1] = interp_pairs<DIM>(sP + stride, SX, SY, nd[0], hf[1], nd[2]);
    e[2] = interp_pairs<DIM>(sP + 2 * stride, SX, SY, nd[0], nd[1], hf[2]);
    b[0] = interp_pairs<DIM>(sP + 3 * stride, SX, SY, nd[0], hf[1], hf[2]);
    b[1] = interp_pairs<DIM>(sP + 4 * stride, SX, SY, hf[0], nd[1], hf[2]);
    b[2] = interp_pairs<DIM>(sP + 5 * stride, SX, SY, hf[0], hf[1], nd[2]);
}

// gather, Boris push and deposit of one particle, FP32 arithmetic, linear shapes
template <int DIM, class SV, class SPV>
__device__ __forceinline__ void push_one_f32lin(const SV& S, const SPV& sp, const Tile& tl,
                                                const float* __restrict__ sEB, const JView& V,
                                                double* __restrict__ sQw, unsigned* s_tail, const SmemPlan& P,
                                                const float* jf, const float* dtd, float kq, float qs,
                                                int64_t p, const PIn& in, int32_t* err) {
    using A = Arith<float>;
    const double Xs[3] = {in.X, DIM == 3 ? in.Y : 0.0, in.Z};
    long long b0[3];
    int c[3];
    float f[3];
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) {
            b0[a] = 0;
            c[a] = 0;
            f[a] = 0.0f;
            continue;
        }
        b0[a] = fix24(Xs[a]);
        c[a] = (int)(b0[a] >> 24) - tl.o[a];
        f[a] = frac24(b0[a]);
        inside = inside && (unsigned)c[a] < (unsigned)S.T[a];
    }
    if (!inside) {
        atomicOr(err, PIC_DERR_BOUNDS);
        sp.key[p] = S.ntiles;
        warp_hist_add(sp.count, S.ntiles);
        return;
    }
    // node supports (start c, weight f of the upper node) and half-node ones
    Support<1, float> nd[3], hf[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) {
            nd[1].s = -1;
            nd[1].w[0] = 1.0f;
            nd[1].w[1] = 0.0f;
            hf[1] = nd[1];
            continue;
        }
        nd[a].s = c[a];
        nd[a].w[1] = f[a];
        const bool up = f[a] >= 0.5f;
        if (S.ec) {
            hf[a].s = c[a];
            hf[a].w[1] = 0.0f;
        } else {
            hf[a].s = up ? c[a] : c[a] - 1;
            hf[a].w[1] = f[a] + (up ? -0.5f : 0.5f);
        }
    }
    float ev[3], bv[3];
    gather6_pairs<DIM>(reinterpret_cast<const float2*>(sEB), P.eb_stride, S.ebs[0], S.ebs[1], nd, hf, ev, bv);
    const float u0 = f32_of(in.u0), u1 = f32_of(in.u1), u2 = f32_of(in.u2);
    const float qw = qs * f32_of(in.w);

    // relativistic Boris push
    const float m0 = fmaf(kq, ev[0], u0), m1 = fmaf(kq, ev[1], u1), m2 = fmaf(kq, ev[2], u2);
    const float ig = rsqrtf(fmaf(m2, m2, fmaf(m1, m1, fmaf(m0, m0, 1.0f))));
    const float kg = kq * ig;
    const float t0 = kg * bv[0], t1 = kg * bv[1], t2 = kg * bv[2];
    const float sf = 2.0f * __frcp_rn(1.0f + fmaf(t2, t2, fmaf(t1, t1, t0 * t0)));
    const float s0 = sf * t0, s1 = sf * t1, s2 = sf * t2;
    const float d0 = fmaf(m1, t2, fmaf(-m2, t1, m0));
    const float d1 = fmaf(m2, t0, fmaf(-m0, t2, m1));
    const float d2 = fmaf(m0, t1, fmaf(-m1, t0, m2));
    const float p0 = fmaf(d1, s2, fmaf(-d2, s1, m0));
    const float p1 = fmaf(d2, s0, fmaf(-d0, s2, m1));
    const float p2 = fmaf(d0, s1, fmaf(-d1, s0, m2));
    const float n0 = fmaf(kq, ev[0], p0), n1 = fmaf(kq, ev[1], p1), n2 = fmaf(kq, ev[2], p2);
    const float ign = rsqrtf(fmaf(n2, n2, fmaf(n1, n1, fmaf(n0, n0, 1.0f))));
    const float v1 = n1 * ign;
    const float dv[3] = {(n0 * ign) * dtd[0], DIM == 3 ? v1 * dtd[1] : 0.0f, (n2 * ign) * dtd[2]};

    // x^{n+1} in the same fixed point; in-cell test and displacement
    long long b1[3];
    float disp[3];
    bool same = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (DIM == 2 && a == 1) {
            b1[a] = 0;
            disp[a] = 0.0f;
            continue;
        }
        const int di = __float2int_rn(dv[a] * 16777216.0f);
        b1[a] = b0[a] + di;
        disp[a] = (float)di * 5.9604644775390625e-8f;
        same = same && (b1[a] >> 24) == (b0[a] >> 24);
    }
    if (same) {
        deposit_lin_incell_d<float, DIM, SV>(S, V, qw, v1, jf, nd, disp);
    } else {
        const unsigned slot = atomicAdd(s_tail, 1u) & (WQ - 1);
        sQw[0 * WQ + slot] = Xs[0];
        sQw[1 * WQ + slot] = Xs[2];
        sQw[2 * WQ + slot] = unfix24(b1[0]);
        sQw[3 * WQ + slot] = unfix24(b1[2]);
        sQw[4 * WQ + slot] = f64_of(qw);
        sQw[5 * WQ + slot] = DIM == 3 ? Xs[1] : f64_of(v1);
        if (DIM == 3) sQw[6 * WQ + slot] = unfix24(b1[1]);
    }

    // new position, boundary, re-sort key
    double X = unfix24(b1[0]), Y = DIM == 3 ? unfix24(b1[1]) : 0.0, Z = unfix24(b1[2]);
    int g[3] = {(int)(b1[0] >> 24), DIM == 3 ? (int)(b1[1] >> 24) : 0, (int)(b1[2] >> 24)};
    const int rel[3] = {g[0] - tl.o[0], g[1] - tl.o[1], g[2] - tl.o[2]};
    if (g[0] < 0 || g[0] >= S.n[0]) {
        X = wrap_periodic(X, S.nd[0]);
        g[0] += g[0] < 0 ? S.n[0] : -S.n[0];
    }
    if (DIM == 3 && (g[1] < 0 || g[1] >= S.n[1])) {
        Y = wrap_periodic(Y, S.nd[1]);
        g[1] += g[1] < 0 ? S.n[1] : -S.n[1];
    }
    int key = -1;
    if (S.absorb > 0) {
        if (g[2] < S.absorb || g[2] >= S.n[2] - S.absorb) key = S.ntiles;
    } else if (g[2] < 0 || g[2] >= S.n[2]) {
        Z = wrap_periodic(Z, S.nd[2]);
        g[2] += g[2] < 0 ? S.n[2] : -S.n[2];
    }
    if (key < 0) {
        key = near_key<DIM>(S, S.nk, rel);
        if (key < 0)
            key = tile_key(S, min(max(g[0], 0), S.n[0] - 1), DIM == 3 ? min(max(g[1], 0), S.n[1] - 1) : 0,
                           min(max(g[2], 0), S.n[2] - 1));
    }
    sp.dst[0][p] = X;
    if (DIM == 3) sp.dst[1][p] = Y;
    sp.dst[2][p] = Z;
    sp.dst[3][p] = f64_of(n0);
    sp.dst[4][p] = f64_of(n1);
    sp.dst[5][p] = f64_of(n2);
    sp.key[p] = key;
    warp_hist_add(sp.count, key);
}

// A warp deposits n <= 32 queued (cell-crossing) particles of its ring,
// starting at slot head, on the ORDER + 2 window: lane i takes entry head + i.
// Supports are taken relative to the origin of tile tl and the view V is that
// tile's; with the global J target any tile gives the same global nodes (the
// entries hold global positions), so rings then drain across tile changes.
template <class R, int DIM, int ORDER>
__device__ __forceinline__ void drain_warp(const SimDev& S, const Tile& tl,
                                           const JView& V,
                                           const double* __restrict__ sQw, unsigned head, unsigned n,
                                           const R* jf, int32_t* err) {
    using A = Arith<R>;
    const unsigned lane = threadIdx.x & 31u;
    if (lane >= n) return;
    const unsigned i = (head + lane) & (WQ - 1);
    const double X = sQw[0 * WQ + i], Z = sQw[1 * WQ + i];
    const double X1 = sQw[2 * WQ + i], Z1 = sQw[3 * WQ + i], qw = sQw[4 * WQ + i];
    const double Y = DIM == 3 ? sQw[5 * WQ + i] : 0.0, vy = DIM == 3 ? 0.0 : sQw[5 * WQ + i];
    const double Y1 = DIM == 3 ? sQw[6 * WQ + i] : 0.0;
    Support<ORDER, R> nd[3], mv[3];
    nd[0] = support_at<ORDER, R>(X, tl.o[0]);
    nd[2] = support_at<ORDER, R>(Z, tl.o[2]);
    mv[0] = support_at<ORDER, R>(X1, tl.o[0]);
    mv[2] = support_at<ORDER, R>(Z1, tl.o[2]);
    if (DIM == 3) {
        nd[1] = support_at<ORDER, R>(Y, tl.o[1]);
        mv[1] = support_at<ORDER, R>(Y1, tl.o[1]);
    } else {
        nd[1].s = -1;
        nd[1].w[0] = A::c(1.0);
        mv[1] = nd[1];
    }
    if (!deposit<R, DIM, ORDER, ORDER + 2>(S, V, A::from(qw), A::from(vy), jf, nd[0], nd[1], nd[2],
                                           mv[0], mv[1], mv[2]))
        atomicOr(err, PIC_DERR_BOUNDS);
}

// the same in FP64, fixed-point: lane i takes entry first + i of the stacks;
// ONE: particles that cross in one direction
template <int DIM, int ORDER, bool ONE>
__device__ __noinline__ void drain_warp_q(const SimDev& S, const Tile& tl, const JView& V,
                                          const double* __restrict__ sQw, unsigned first, unsigned n,
                                          int32_t* err) {
    const unsigned lane = threadIdx.x & 31u;
    if (lane >= n) return;
    const unsigned i = first + lane;
    const double x0[3] = {sQw[0 * QSLOTS + i], DIM == 3 ? sQw[5 * QSLOTS + i] : 0.0, sQw[1 * QSLOTS + i]};
    const double x1[3] = {sQw[2 * QSLOTS + i], DIM == 3 ? sQw[6 * QSLOTS + i] : 0.0, sQw[3 * QSLOTS + i]};
    const double qw = sQw[4 * QSLOTS + i], vy = DIM == 3 ? 0.0 : sQw[5 * QSLOTS + i];
    const Amp ja[3] = {amp_of(S.jfac[0]), amp_of(DIM == 3 ? S.jfac[1] : S.jyfac2d), amp_of(S.jfac[2])};
    bool ok;
    if (amps_safe<DIM>(exp_range(S.jfac[0], DIM == 3 ? S.jfac[1] : S.jyfac2d, S.jfac[2]), qw, vy)) {
        SupQ<ORDER> nd[3], mv[3];
        bool nan = false;  // a NaN position comes with a NaN qw, which is not safe
        node_supports_q<DIM, ORDER>(x0, tl.o, nd, nan);
        node_supports_q<DIM, ORDER>(x1, tl.o, mv, nan);
        if constexpr (ONE) {
            const int a = nd[0].s != mv[0].s ? 0 : (DIM == 3 && nd[1].s != mv[1].s ? 1 : 2);
            // a move of more than one node is out of bounds
            const int step = pick3(a, mv[0].s, mv[1].s, mv[2].s) - pick3(a, nd[0].s, nd[1].s, nd[2].s);
            ok = step == 1 || step == -1;
            if (ok) deposit_one_axis<DIM, ORDER>(S.jlo, V, ja, qw, vy, nd, mv, a);
        } else {
            ok = deposit_q<DIM, ORDER, ORDER + 2, false>(S.jlo, V, ja, nullptr, qw, vy, nd, mv);
        }
    } else {
        ok = deposit_any<DIM, ORDER>(S, V, tl.o[0], tl.o[1], tl.o[2], x0[0], x0[1], x0[2], x1[0], x1[1], x1[2], qw, vy);
    }
    if (!ok) atomicOr(err, PIC_DERR_BOUNDS);
}

// the J view of tile tl: the global padded arrays
__device__ __forceinline__ JView j_view(const SimDev& S, const Tile& tl) {
    JView v;
    const int lo = S.jlo;
    v.base = S.F[6] + pidx(S, tl.o[0] - lo, S.dim == 3 ? tl.o[1] - lo : 0, tl.o[2] - lo);
    v.cs = (int64_t)S.pn[0] * S.pn[1] * S.pn[2];
    v.sy = S.pn[0];
    v.sz = S.pn[0] * S.pn[1];
    return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// the simulation's constants in the push arithmetic R
template <class R, int DIM>
struct SimConsts {
    R jf[3], dtd[3];
    __device__ __forceinline__ explicit SimConsts(const SimDev& S) {
        using A = Arith<R>;
        jf[0] = A::from(S.jfac[0]);
        jf[1] = A::from(DIM == 3 ? S.jfac[1] : S.jyfac2d);
        jf[2] = A::from(S.jfac[2]);
        dtd[0] = A::from(S.dtd[0]);
        dtd[1] = A::from(S.dtd[1]);
        dtd[2] = A::from(S.dtd[2]);
    }
};

// MINB = resident CTAs per SM the register allocation is sized for (1: up to
// 255 registers, 8 warps per SM; 2: at most 128 registers, 16 warps per SM).
// PREC = arithmetic of the particle push: 0 FP64, 2 FP32 (storage,
// positions and index math stay FP64 in both, and the current goes to the
// global FP64 J by L2 reductions).
// PPT = particles per thread per loop iteration: their HBM loads are issued
// together before the first of them is pushed (with PPT 1 each lane's
// next particle is staged through shared memory instead).
template <int DIM, int ORDER, int MINB, int PREC, int PPT>
__global__ void __launch_bounds__(256, MINB) pic_particle_kernel(const SchedDev* __restrict__ sd,
                                                              SimDev* __restrict__ sims) {
    using R = typename std::conditional<PREC == 2, float, double>::type;
    using A = Arith<R>;
    extern __shared__ __align__(128) double smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    // TMA destinations must be 128-byte aligned: round the dynamic base up
    double* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 127u) / sizeof(double);
    __shared__ int s_unit, s_list, s_abort, s_tile0, s_tile1;
    __shared__ HotSim s_hot;
    __shared__ unsigned s_qhead[QMAXWARPS], s_qtail[QMAXWARPS];
    __shared__ unsigned long long s_cost, s_time;
    __shared__ int s_emax[6];  // fixed-point tile: biased exponent of each component's largest magnitude
    __shared__ int s_emin[6];  // and of its weakest place (scan_tile)
    __shared__ int s_some;     // whether a cell is marked as too weak for it (mark_weak)

    const int nlists = sd->meta[0];
    const int steal = sd->meta[1];
    const int my_list = blockIdx.x % nlists;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        s_list = my_list;
        s_abort = 0;
        for (int w = 0; w < QMAXWARPS; ++w) s_qhead[w] = s_qtail[w] = 0u;
        s_cost = s_time = 0ull;
    }
    __syncthreads();
    uint32_t phase = 0;
    Tile cur;
    cur.sim = -1;
    cur.t = -1;
    int visited = 0, hot = -1;
    const unsigned* weak = nullptr;  // the marks, if the staged tile has such cells
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // ring of cell-crossing particles, in global scratch (L1/L2 resident; a
    // drain runs once per 32 crossings)
    double* const gring = sd->rings + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * PIC_RING_DOUBLES;

    // Drains the warp's crossing particles: groups of 32 while that many wait,
    // or (all) everything.  They outlive tile changes (with the global J every
    // tile gives the same global nodes) and are drained completely when the
    // simulation changes (they are one simulation's) and at the end.
    auto drain = [&](const SimDev& CS, const JView& V, const R* jf, bool all) {
        __syncwarp();
        if constexpr (PREC == 2) {
            const unsigned head = s_qhead[warp], wait = *(volatile unsigned*)(s_qtail + warp) - head;
            const unsigned n = wait >= 32u ? 32u : (all ? wait : 0u);
            if (n > 0u) {
                drain_warp<R, DIM, ORDER>(CS, cur, V, gring, head, n, jf, sd->err);
                __syncwarp();
                if (lane == 0) s_qhead[warp] = head + n;
                __syncwarp();
            }
        } else {
            const unsigned one = *(volatile unsigned*)(s_qtail + warp), many = *(volatile unsigned*)(s_qhead + warp);
            const unsigned n1 = one >= 32u ? 32u : (all ? one : 0u), nm = many >= 32u ? 32u : (all ? many : 0u);
            if constexpr (ORDER > 1)
                if (n1 > 0u) drain_warp_q<DIM, ORDER, true>(CS, cur, V, gring, one - n1, n1, sd->err);
            if (nm > 0u) drain_warp_q<DIM, ORDER, false>(CS, cur, V, gring, QSLOTS - many, nm, sd->err);
            if (n1 + nm > 0u) {
                __syncwarp();
                if (lane == 0) {
                    s_qtail[warp] = one - n1;
                    s_qhead[warp] = many - nm;
                }
                __syncwarp();
            }
        }
    };
    auto drain_all = [&](const SimDev& CS) {
        const SimConsts<R, DIM> K(CS);
        drain(CS, j_view(CS, cur), K.jf, true);
        if (PREC == 2) drain(CS, j_view(CS, cur), K.jf, true);  // up to 63 wait
    };

    while (true) {
        if (threadIdx.x == 0) {
            int u = -1;
            while (visited < nlists) {
                int L = s_list;
                int pos = atomicAdd(sd->head + L, 1);
                int b = sd->list_off[L], e = sd->list_off[L + 1];
                if (b + pos < e) { u = b + pos; break; }
                if (!steal) { visited = nlists; break; }
                s_list = (L + 1) % nlists;
                ++visited;
            }
            s_unit = u;
            s_tile0 = 0x7FFFFFFF;
            s_tile1 = -1;
        }
        __syncthreads();
        const int u = s_unit;
        if (u < 0) break;
        const UnitDev unit = sd->units[u];
        const SimDev& S = sims[unit.sim];
        const bool cap_clk = (S.capture & 1) != 0, cap_time = (S.capture & 2) != 0;
        const SmemPlan P = smem_plan(S.ebs);
        double* sEBd = smem;
        unsigned* const s_bits = reinterpret_cast<unsigned*>(smem + P.bit_off);
        const R* sEB = reinterpret_cast<const R*>(smem);
        unsigned long long my_clk = 0ull;
        const SimConsts<R, DIM> K(S);
        const int t_first = unit.box * S.tiles_per_box;
        const int t_end = t_first + S.tiles_per_box;

        // the unit's particle range of each species, and the tiles it touches
        if (unit.sim != hot) {
            stage_hot(s_hot, S);
            hot = unit.sim;
        }
        {
            const int i = (int)threadIdx.x - 4;
            if (i >= 0 && i < S.nsp) {
                const SpeciesDev& sp = S.sp[i];
                const int64_t b0 = sp.off[t_first], nbp = sp.off[t_end] - b0;
                s_hot.sp[i].r0 = b0 + (nbp * unit.chunk) / unit.nchunks;
                s_hot.sp[i].r1 = b0 + (nbp * (unit.chunk + 1)) / unit.nchunks;
            }
        }
        __syncthreads();
        const int nsp = s_hot.nsp;
        for (int i = threadIdx.x; i < nsp * S.tiles_per_box; i += blockDim.x) {
            const int spi = i / S.tiles_per_box, t = t_first + i - spi * S.tiles_per_box;
            const HotSp& sp = s_hot.sp[spi];
            if (max(sp.off[t], sp.r0) < min(sp.off[t + 1], sp.r1)) {
                atomicMin(&s_tile0, t);
                atomicMax(&s_tile1, t);
            }
        }
        __syncthreads();
        uint64_t my_ns = 0ull;  // lane 0: ns of this warp's particle loops
        // tile by tile, the species inside: a tile is staged once for all of them
        {
            const int t1 = s_tile1;
            for (int t = s_tile0; t <= t1; ++t) {
                bool any = false;
                for (int spi = 0; spi < nsp; ++spi) {
                    const HotSp& sp = s_hot.sp[spi];
                    any = any || max(sp.off[t], sp.r0) < min(sp.off[t + 1], sp.r1);
                }
                if (!any) continue;
                if (t != cur.t || unit.sim != cur.sim) {
                    if (cur.t >= 0 && unit.sim != cur.sim) drain_all(sims[cur.sim]);
                    __syncthreads();
                    cur.sim = unit.sim;
                    cur.t = t;
                    tile_origin(S, t, cur.o);
                    if (threadIdx.x == 0) {
                        for (int c = 0; c < 6; ++c) {
                            s_emax[c] = 0;
                            s_emin[c] = 0x7FFF;
                        }
                        s_some = 0;
                        fence_proxy_async();
                        mbar_expect_tx(&bar, (uint32_t)(6 * P.eb_vol * sizeof(double)));
                        constexpr int H = EBHalo<ORDER>::lo;
                        const int x0 = cur.o[0] - H + S.g[0];
                        const int y0 = (DIM == 3) ? cur.o[1] - H + S.g[1] : 0;
                        const int z0 = cur.o[2] - H + S.g[2];
#pragma unroll
                        for (int c = 0; c < 6; ++c)
                            tma_load_3d(sEBd + c * P.eb_stride, &S.tmap[c], x0, y0, z0, &bar);
                    }
                    for (int i = threadIdx.x; i < 9; i += blockDim.x) {
                        const int a = i / 3, side = i - 3 * a;
                        const int c = a == 0 ? cur.o[0] : (a == 1 ? cur.o[1] : cur.o[2]);
                        s_hot.nk[a][side] = DIM == 2 && a == 1 ? 0 : key_part(s_hot, a, side == 0 ? c - 1 : (side == 1 ? c : c + s_hot.T[a]));
                    }
                    bool ok = mbar_wait_bounded(&bar, phase);
                    phase ^= 1u;
                    if (!ok) {
                        atomicOr(sd->err, PIC_DERR_TMA_TIMEOUT);
                        atomicExch(&s_abort, 1);
                    }
                    __syncthreads();
                    if (s_abort) {
                        // the copies may still be in flight: one more bounded wait, then leave
                        if (threadIdx.x == 0) mbar_wait_bounded(&bar, phase ^ 1u);
                        __syncthreads();
                        return;
                    }
                    if constexpr (PREC != 2) {
                        // E/B tile to fixed point in place: the exponent of each
                        // component's largest magnitude, then the values in its units
                        scan_tile<ORDER>(sEBd, P.eb_stride, P.eb_vol, S.ec != 0, s_emax, s_emin);
                        __syncthreads();
                        bool fx = true, some = false;
                        for (int c = 0; c < 6; ++c) {
                            const int em = s_emax[c];
                            fx = fx && tile_exp_ok(em);
                            some = some || (em != 0 && s_emin[c] < (int)weak_limit<ORDER>(em));
                        }
                        if (fx) {
                            if (some && mark_weak<ORDER, DIM>(s_bits, P.bit_words, sEBd, P.eb_stride, P.eb_vol, S.ebs[0],
                                                              S.ebs[1], s_emax, S.ec != 0))
                                s_some = 1;
                        } else {  // every cell: Inf, NaN, or magnitudes outside the exponent range
                            for (int i = threadIdx.x; i < 6 * P.bit_words; i += blockDim.x) s_bits[i] = ~0u;
                            s_some = 1;
                        }
                        if (some) __syncthreads();  // (marked before it is converted)
                        if (fx) {
                            for (int c = 0; c < 6; ++c) {
                                const int em = s_emax[c];
#pragma unroll 4
                                for (int i = threadIdx.x; i < P.eb_vol; i += blockDim.x) {
                                    double* v = sEBd + c * P.eb_stride + i;
                                    *v = __longlong_as_double(tile_fix<TileBits<ORDER>::FB>(*v, em));
                                }
                            }
                        }
                        __syncthreads();
                        weak = s_some ? s_bits : nullptr;
                    }
                    if constexpr (PREC == 2) {
                        // E/B tile to FP32 in place, in rounds of 8 elements per thread
                        // (nt threads); round m reads doubles [8 nt m, 8 nt (m + 1)] and,
                        // after its barrier, writes elements [8 nt m, 8 nt (m + 1)).
                        // Linear shapes: element i becomes the float pair (F[i],
                        // F[i+1] - F[i]) in the 8 bytes of double i (the pair at the end
                        // of a row is never read).  Other orders: element i becomes float
                        // i, overlaying doubles [4 nt m, 4 nt (m + 1)).  Either way a
                        // round writes only doubles read by rounds <= m and none read by a
                        // later round.
                        const int ntot = 6 * P.eb_stride, nt = blockDim.x;
                        for (int r0 = 0; r0 < ntot; r0 += 8 * nt) {
                            float v[8], d[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const int i = r0 + k * nt + threadIdx.x;
                                v[k] = i < ntot ? f32_of(sEBd[i]) : 0.0f;
                                if constexpr (ORDER == 1) d[k] = i + 1 < ntot ? f32_of(sEBd[i + 1]) - v[k] : 0.0f;
                            }
                            __syncthreads();
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const int i = r0 + k * nt + threadIdx.x;
                                if (i < ntot) {
                                    if constexpr (ORDER == 1)
                                        reinterpret_cast<float2*>(sEBd)[i] = make_float2(v[k], d[k]);
                                    else
                                        reinterpret_cast<float*>(sEBd)[i] = v[k];
                                }
                            }
                        }
                        __syncthreads();
                    }
                }
                const uint64_t t0 = lane == 0 && cap_time ? globaltimer() : 0ull;
                const unsigned long long c0 = cap_clk ? clock64() : 0ull;
                // groups of particles go round the warps, on across the species
                const int nw = blockDim.x >> 5;
                int turn = warp;
                for (int spi = 0; spi < nsp; ++spi) {
                    // per-warp loop: no CTA barrier until the tile changes
                    const HotSp& hs = s_hot.sp[spi];
                    const int64_t s0 = max(hs.off[t], hs.r0), s1 = min(hs.off[t + 1], hs.r1);
                    if (s0 >= s1) continue;
                    const R kq = A::from(hs.kq);
                    const R qs = A::from(hs.q);
                    const double qsd = hs.q;
                    const int64_t first = s0 + turn * (32 * PPT);
                    {
                        // this warp's place in the round after the species' last group
                        const int ng = (int)((s1 - s0 + 32 * PPT - 1) / (32 * PPT));
                        turn = (turn - ng) % nw;
                        if (turn < 0) turn += nw;
                    }
                    const JView V = j_view(S, cur);
                    double* sQw = gring;
                    const int64_t* const order = PREC == 2 ? hs.order : nullptr;  // (FP32 alone steps indirectly)
                    auto place = [&](int64_t p) {
                        if (!order) return p;
                        // (a step that gave up on a tile load leaves places unset)
                        const int64_t o = order[p];
                        return (uint64_t)o < (uint64_t)hs.cap ? o : p;
                    };
                    auto push = [&](int64_t p, int64_t src, const PIn& in) {
                        // an indirect push carries the weight and the id along
                        const int64_t id = order ? hs.id_src[src] : 0;
                        if constexpr (PREC != 2)
                            push_one_q<R, DIM, ORDER>(s_hot, s_hot.sp[spi], S, cur, sEBd, weak, s_emax, V, sQw,
                                                      s_qtail + warp, s_qhead + warp, P, K.dtd, kq, qsd, p, in,
                                                      sd->err);
                        else if constexpr (ORDER == 1)
                            push_one_f32lin<DIM>(s_hot, s_hot.sp[spi], cur, sEB, V, sQw, s_qtail + warp, P, K.jf,
                                                 K.dtd, kq, qs, p, in, sd->err);
                        else
                            push_one<R, DIM, ORDER>(s_hot, s_hot.sp[spi], cur, sEB, V, sQw, s_qtail + warp, P,
                                                    K.jf, K.dtd, kq, qs, p, in, sd->err);
                        if (order) {
                            hs.dst[6][p] = in.w;
                            hs.id_dst[p] = id;
                        }
                    };
                    auto drain_full = [&]() { drain(S, V, K.jf, false); };
                    if constexpr (PPT == 1) {
                        // the particle loads are a latency the loop waits on; each
                        // lane stages its next particle into shared memory with cp.async
                        // one iteration ahead (two buffers per warp, the lane's own column)
                        double* const pbw = smem + P.pb_off + warp * (2 * PIN_SLOTS) + lane;
                        // (indirect: its place is read one iteration before that)
                        const int64_t bd = blockDim.x, pf = first + lane;
                        int64_t src = pf < s1 ? place(pf) : 0, nxt = pf + bd < s1 ? place(pf + bd) : 0;
                        if (P.staged && pf < s1) stage_in<DIM>(hs, src, pbw);
                        cp_async_commit();
                        unsigned buf = 0u;
                        for (int64_t p0 = first; p0 < s1; p0 += bd) {
                            const int64_t p = p0 + lane;
                            if (P.staged && p + bd < s1) stage_in<DIM>(hs, nxt, pbw + (buf ^ 1u) * PIN_SLOTS);
                            cp_async_commit();
                            const int64_t after = p + 2 * bd < s1 ? place(p + 2 * bd) : 0;
                            cp_async_wait<1>();
                            if (p < s1)
                                push(p, src, P.staged ? read_staged<DIM>(pbw + buf * PIN_SLOTS) : load_one<DIM>(hs, src));
                            src = nxt;
                            nxt = after;
                            buf ^= 1u;
                            drain_full();
                        }
                        cp_async_wait<0>();
                    } else {
                        for (int64_t p0 = first; p0 < s1; p0 += (int64_t)blockDim.x * PPT) {
                            PIn in[PPT];
                            int64_t src[PPT];
#pragma unroll
                            for (int q = 0; q < PPT; ++q) {
                                const int64_t p = p0 + q * 32 + lane;
                                if (p < s1) {
                                    src[q] = place(p);
                                    in[q] = load_one<DIM>(hs, src[q]);
                                }
                            }
#pragma unroll
                            for (int q = 0; q < PPT; ++q) {
                                const int64_t p = p0 + q * 32 + lane;
                                if (p < s1) push(p, src[q], in[q]);
                                drain_full();
                            }
                        }
                    }
                    __syncwarp();
                }
                if (cap_clk) my_clk += clock64() - c0;
                if (lane == 0 && cap_time) my_ns += globaltimer() - t0;
            }
        }
        // in-situ cost: thread clocks -> warp sum -> shared -> one global add per unit
        if (cap_clk) {
            unsigned long long ws = warp_sum_u64(my_clk);
            if ((threadIdx.x & 31) == 0 && ws) atomicAdd(&s_cost, ws);
        }
        if (lane == 0 && my_ns) atomicAdd(&s_time, (unsigned long long)my_ns);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_cost) atomicAdd((unsigned long long*)(S.cost_clock + unit.box), s_cost);
            s_cost = 0ull;
            // kernel-time cost: span of the unit's particle loops, the mean over the
            // CTA's warps (a unit that fills them is charged its wall time, one that
            // leaves warps idle the share it uses)
            if (cap_time)
                atomicAdd((unsigned long long*)(S.cost_time + unit.box), s_time / (unsigned long long)(blockDim.x >> 5));
            s_time = 0ull;
        }
    }
    if (cur.t >= 0) drain_all(sims[cur.sim]);
}

// ---- host side of one precision: launch, attributes, occupancy
template <int DIM, int ORDER, int PREC>
static cudaError_t launch_particles_t(const LaunchCfg& cfg, size_t smem, const SchedDev* sched,
                                      SimDev* sims, cudaStream_t st) {
    const bool two = cfg.ppt == 2;
    if (cfg.minb == 2) {
        if (two) pic_particle_kernel<DIM, ORDER, 2, PREC, 2><<<cfg.ctas, cfg.threads, smem, st>>>(sched, sims);
        else pic_particle_kernel<DIM, ORDER, 2, PREC, 1><<<cfg.ctas, cfg.threads, smem, st>>>(sched, sims);
    } else {
        if (two) pic_particle_kernel<DIM, ORDER, 1, PREC, 2><<<cfg.ctas, cfg.threads, smem, st>>>(sched, sims);
        else pic_particle_kernel<DIM, ORDER, 1, PREC, 1><<<cfg.ctas, cfg.threads, smem, st>>>(sched, sims);
    }
    return cudaGetLastError();
}

template <class K>
static cudaError_t set_smem(K kernel, size_t smem) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <int DIM, int ORDER, int PREC>
static cudaError_t prepare_t(size_t smem) {
    cudaError_t e = set_smem(pic_particle_kernel<DIM, ORDER, 1, PREC, 1>, smem);
    if (e == cudaSuccess) e = set_smem(pic_particle_kernel<DIM, ORDER, 2, PREC, 1>, smem);
    if (e == cudaSuccess) e = set_smem(pic_particle_kernel<DIM, ORDER, 1, PREC, 2>, smem);
    if (e == cudaSuccess) e = set_smem(pic_particle_kernel<DIM, ORDER, 2, PREC, 2>, smem);
    return e;
}

template <int DIM, int ORDER, int PREC>
static int occupancy_t(int minb, int ppt, int threads, size_t smem) {
    int n = 0;
    cudaError_t e;
    if (minb == 2)
        e = ppt == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pic_particle_kernel<DIM, ORDER, 2, PREC, 2>,
                                                                     threads, smem)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pic_particle_kernel<DIM, ORDER, 2, PREC, 1>,
                                                                     threads, smem);
    else
        e = ppt == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pic_particle_kernel<DIM, ORDER, 1, PREC, 2>,
                                                                     threads, smem)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pic_particle_kernel<DIM, ORDER, 1, PREC, 1>,
                                                                     threads, smem);
    return e == cudaSuccess ? n : 0;
}

// dispatch over the shape order for one precision (PIC_PREC) and one
// dimensionality (PIC_DIM): each translation unit instantiates one pair
#define PIC_DISPATCH_DO(FN, ...)                                            \
    do {                                                                    \
        if (order == 1) return FN<PIC_DIM, 1, PIC_PREC>(__VA_ARGS__);       \
        if (order == 2) return FN<PIC_DIM, 2, PIC_PREC>(__VA_ARGS__);       \
        if (order == 3) return FN<PIC_DIM, 3, PIC_PREC>(__VA_ARGS__);       \
    } while (0)

}  // namespace

// the three entry points of one translation unit, suffix SUF = p<prec>_d<dim>
#define PIC_DEFINE_PARTICLE_TU(SUF)                                                                      \
    cudaError_t pic_launch_particles_##SUF(int order, const LaunchCfg& cfg, size_t smem,                 \
                                           const SchedDev* sched, SimDev* sims, cudaStream_t st) {       \
        PIC_DISPATCH_DO(launch_particles_t, cfg, smem, sched, sims, st);                                  \
        return cudaErrorInvalidValue;                                                                     \
    }                                                                                                     \
    cudaError_t pic_prepare_particles_##SUF(int order, size_t smem) {                                     \
        PIC_DISPATCH_DO(prepare_t, smem);                                                                 \
        return cudaErrorInvalidValue;                                                                     \
    }                                                                                                     \
    int pic_particle_occupancy_##SUF(int order, int minb, int ppt, int threads, size_t smem) {            \
        PIC_DISPATCH_DO(occupancy_t, minb, ppt, threads, smem);                                           \
        return 0;                                                                                         \
    }
