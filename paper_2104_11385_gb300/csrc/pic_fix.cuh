// pic_fix.cuh -- 64-bit fixed-point arithmetic of the particle kernel's field
// gather and current deposit.
//
// GB300 issues one FP64 warp instruction per SM every 16 clocks (2 lanes per
// SM per clock), against 4 integer warp instructions per clock.  The gather
// and the deposit work on quantities of known range: B-spline weights and
// in-cell offsets lie in [0, 1], and the fields a particle sees are bounded by
// the largest magnitude of its staged tile.  They are therefore held as 64-bit
// integers and multiplied with three or four 32x32->64-bit IMADs each, which
// keeps more bits than FP64 does (about 60 against 53) and leaves the FP64 pipe
// to the Boris push:
//   Q62     a weight, an offset or a move in cells, in units of 2^-62
//   tile    a field value in units of 2^(e - FB), 2^e > every magnitude of that
//           component in the tile; FB = 62 for linear shapes, 60 for the
//           others (headroom of the row sums).  A value down to 2^-9 (2^-7) of
//           the largest keeps a double's 53 bits, a smaller one fewer: the tile's
//           places where a component is weak are marked when it is staged
//           (weak_limit), and their particles gather it by itself
//   Amp     a floating-point factor: 64-bit mantissa, exponent, sign
// Only the last step of each chain returns to IEEE doubles, by bit operations
// and with one rounding: the six field values, and every current contribution.
#pragma once
#include <cuda_runtime.h>

namespace {

typedef long long q62;           // signed, units of 2^-62
typedef unsigned long long u64;

// 32 x 32 -> 64-bit products, and the same added to c.  In PTX: from the C
// expressions the compiler widens the operands that come out of a 64-bit
// subtraction or shift and multiplies 64 x 64 bits (20 instructions for a lerp
// instead of 9).
__device__ __forceinline__ long long mul_ss(int a, int b) {
#ifdef __CUDA_ARCH__
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (long long)a * b;
#endif
}
__device__ __forceinline__ long long mad_ss(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (long long)a * b + c;
#endif
}
__device__ __forceinline__ u64 mul_uu(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (u64)a * b;
#endif
}
__device__ __forceinline__ u64 mad_uu(unsigned a, unsigned b, u64 c) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (u64)a * b + c;
#endif
}

constexpr q62 kOneQ = 1ll << 62;
constexpr q62 kHalfQ = 1ll << 61;

// balanced limbs: v = h 2^32 + l with l in [-2^31, 2^31)
struct Limb {
    int h, l;
};
__device__ __forceinline__ Limb limb_of(q62 v) {
    const int l = (int)v;
    return Limb{(int)(v >> 32) - (l >> 31), l};
}

// a product of two Q62 numbers (|a|, |b| <= 1), or a sum of such products with
// a total of at most 1, in two accumulators: the 2^64 and the 2^32 terms (the
// product of the low limbs, below one unit, is dropped)
struct AccQ {
    long long hi = 0, mid = 0;
    __device__ __forceinline__ void mac(const Limb& a, const Limb& b) {
        hi = mad_ss(a.h, b.h, hi);
        mid = mad_ss(a.h, b.l, mid);
        mid = mad_ss(a.l, b.h, mid);
    }
    // a tile value v times a weight w >= 0: v's low limb stays unsigned
    __device__ __forceinline__ void mac(long long v, const Limb& w) {
        const int vh = (int)(v >> 32);
        hi = mad_ss(vh, w.h, hi);
        mid = mad_ss(vh, w.l, mid);
        mid = (long long)mad_uu((unsigned)v, (unsigned)w.h, (u64)mid);
    }
    __device__ __forceinline__ long long get() const { return (hi << 2) + (mid >> 30); }
};
__device__ __forceinline__ q62 mulq(const Limb& a, const Limb& b) {
    AccQ s;
    s.mid = 1ll << 29;  // to nearest
    s.mac(a, b);
    return s.get();
}
// a + w (b - a), w in [0, 1]; |a|, |b| < 2^62
__device__ __forceinline__ long long lerpq(long long a, long long b, const Limb& w) {
    AccQ s;
    s.mac(b - a, w);
    return a + s.get();
}

// high 64 bits of a product, at most 2 units low; a < 2^63, b < 2^63
__device__ __forceinline__ u64 mulhi(u64 a, u64 b) {
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
    const u64 mid = mad_uu(al, bh, mul_uu(ah, bl));
    return mad_uu(ah, bh, mid >> 32);
}

// v 2^x as an IEEE double, v < 2^63, rounded to nearest (ROUND) or toward zero: hi is the exponent part of
// its high word, (x + 1085) << 20 (with a sign bit, if any); v != 0 or the result
// is meaningless.
template <bool ROUND>
__device__ __forceinline__ double pack_double(u64 v, unsigned hi) {
    unsigned h = (unsigned)(v >> 32), lo = (unsigned)v;
    if (h == 0u) {
        h = lo >> 1;
        lo <<= 31;
        hi -= 31u << 20;
    }
    const int l = __clz((int)h);
    // leading one in bit 62: the half unit that rounds cannot carry out
    const u64 m = ((((u64)__funnelshift_l(lo, h, l - 1) << 32) | (lo << (l - 1))) + (ROUND ? 0x200u : 0u)) >> 10;
    // (53 bits: the leading one adds 1 to the exponent field)
    return __longlong_as_double((long long)(((u64)((unsigned)(m >> 32) + hi - ((unsigned)l << 20)) << 32) | (unsigned)m));
}

// ---- positions: cell and in-cell offset ----------------------------------
struct CellQ {
    int i;
    q62 q;
    bool nan;
};
static __device__ __noinline__ CellQ cell_q_slow(double x) {
    const double fl = floor(x);
    const double f = x - fl;  // in [0, 1]
    return CellQ{(int)fl, __double2ll_rn(f * 4611686018427387904.0), !(x == x)};
}
// floor(x) and x - floor(x) (below 2^-62 of a cell truncated) by integer work
// for 2^-10 <= x < 2^31; other x go through floor()
__device__ __forceinline__ CellQ cell_q(double x) {
    const u64 b = (u64)__double_as_longlong(x);
    const int e = (int)(b >> 52) - 1023;  // sign set -> e > 1023
    if ((unsigned)(e + 10) <= 40u) {
        const u64 m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
        return CellQ{(int)(m >> (52 - e)), (q62)((m << (e + 10)) & 0x3FFFFFFFFFFFFFFFull), false};
    }
    return cell_q_slow(x);
}

// one-dimensional B-spline support: first node and ORDER + 1 weights (linear:
// only the upper weight w[1] is set)
template <int ORDER>
struct SupQ {
    int s;
    q62 w[ORDER + 1];
};

__device__ __forceinline__ void cubic_weights_q(q62 f, q62* w) {
    // w3 = f^3/6, w1 = 2/3 - f^2 + f^3/2, w0 = (1 - 3f + 3f^2 - f^3)/6, and the sum is 1
    const Limb fl = limb_of(f);
    const q62 f2 = mulq(fl, fl);
    const q62 f3 = mulq(limb_of(f2), fl);
    const q62 w3 = mulq(limb_of(f3), limb_of(768614336404564651ll));  // 2^62 / 6
    const q62 w0 = 768614336404564651ll - (f >> 1) + (f2 >> 1) - w3;
    const q62 w1 = 3074457345618258603ll - f2 + 3 * w3;               // 2^63 / 3
    w[0] = max(w0, 0ll);
    w[1] = w1;
    w[2] = kOneQ - w[0] - w1 - w3;
    w[3] = w3;
}
// quadratic: d = offset from the nearest node, in [-1/2, 1/2]: w0 = (1/2 - d)^2 / 2, w2 = w0 + d
__device__ __forceinline__ void quad_weights_q(q62 d, q62* w) {
    const Limb a = limb_of(kHalfQ - d);
    w[0] = mulq(a, a) >> 1;
    w[2] = max(w[0] + d, 0ll);
    w[1] = kOneQ - w[0] - w[2];
}

// node support of a position
template <int ORDER>
__device__ __forceinline__ SupQ<ORDER> node_support(const CellQ& c, int o) {
    SupQ<ORDER> r;
    if constexpr (ORDER == 1) {
        r.s = c.i - o;
        r.w[1] = c.q;
    } else if constexpr (ORDER == 2) {
        const bool up = c.q >= kHalfQ;
        r.s = c.i - o + (up ? 1 : 0) - 1;
        quad_weights_q(up ? c.q - kOneQ : c.q, r.w);
    } else {
        r.s = c.i - o - 1;
        cubic_weights_q(c.q, r.w);
    }
    return r;
}
// half-node support (the grid shifted by +1/2 cell); ec: the energy-conserving
// one of order ORDER - 1, with a zero last weight
template <int ORDER>
__device__ __forceinline__ SupQ<ORDER> half_support(const CellQ& c, int o, bool ec) {
    SupQ<ORDER> r;
    const bool up = c.q >= kHalfQ;
    const q62 g = up ? c.q - kHalfQ : c.q + kHalfQ;  // offset on the half-node grid
    const int ig = c.i - o - (up ? 0 : 1);
    if constexpr (ORDER == 1) {
        r.s = ec ? c.i - o : ig;
        r.w[1] = ec ? 0 : g;
    } else if constexpr (ORDER == 2) {
        if (ec) {
            r.s = ig;
            r.w[0] = kOneQ - g;
            r.w[1] = g;
            r.w[2] = 0;
        } else {  // nearest half node: floor(x)
            r.s = c.i - o - 1;
            quad_weights_q(c.q - kHalfQ, r.w);
        }
    } else {
        if (ec) {
            r.s = c.i - o - 1;
            quad_weights_q(c.q - kHalfQ, r.w);
            r.w[3] = 0;
        } else {
            r.s = ig - 1;
            cubic_weights_q(g, r.w);
        }
    }
    return r;
}

// ---- tile values ----------------------------------------------------------
template <int ORDER>
struct TileBits {
    static constexpr int FB = ORDER == 1 ? 62 : 60;
};
// biased exponent of the largest magnitude of a component: 0 (all zeros or
// subnormal, held as zero) or within these bounds; a tile outside them (Inf and
// NaN among others) is gathered in FP64
__device__ __forceinline__ bool tile_exp_ok(int e) { return e == 0 || (e >= 128 && e <= 1900); }

// The weakest field that is gathered in fixed point, as a double's exponent: 2^-10
// (linear) or 2^-8 of the component's largest magnitude in the tile.  Error
// of the gather against exact arithmetic, relative to the strongest node it
// interpolates from, random nodes (rms, largest):
//                           linear 3D            cubic 3D
//   nodes near the largest  1.5e-17, 1.0e-16     8.4e-18, 5.7e-17
//   nodes at the limit      1.7e-15, 1.4e-14     1.4e-15, 7.5e-15
//   FP64                    3.7e-17, 3.9e-16     3.7e-17, 3.5e-16
// so a weak place keeps 46 bits or more, and all of them where it is weaker still:
// there a component is gathered by itself, in units of its own nodes' largest.  A
// laser on a foil has whole layers between 2^-7 and 2^-10 behind the skin: limits of
// 2^-7 and 2^-5 cost the 256^3 foil 24 % of its particle kernel there and the cubic
// disk 12 %, 2^-8 and 2^-6 14 % and 4 %, these about 1 %.
template <int ORDER>
__device__ __forceinline__ unsigned weak_limit(int emax) {
    return (unsigned)(emax - (ORDER == 1 ? 10 : 8));
}

// a double in units of 2^(emax - 1022 - FB), rounded to nearest; emax: biased
// exponent of the component's largest magnitude
template <int FB>
__device__ __forceinline__ long long tile_fix(double v, int emax) {
    const u64 b = (u64)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7FFull);
    const u64 m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = e - emax + FB - 53;  // left shift
    u64 f = sh >= 0 ? m << sh : ((m >> min(-sh - 1, 63)) + 1ull) >> 1;
    f = e == 0 ? 0ull : f;
    return (long long)b < 0 ? -(long long)f : (long long)f;
}

// r in units of 2^(emax - 1022 - FB) to double, rounded to nearest; be = emax + 63 - FB
__device__ __forceinline__ double fix_double(long long r, int be) {
    const double v = pack_double<true>((u64)(r < 0 ? -r : r), ((unsigned)be << 20) + ((unsigned)((u64)r >> 32) & 0x80000000u));
    return r == 0ll ? 0.0 : v;
}

template <int ORDER>
struct AxisQ {
    int s;
    Limb w[ORDER + 1];
};
template <int ORDER>
__device__ __forceinline__ AxisQ<ORDER> axis_of(const SupQ<ORDER>& u) {
    AxisQ<ORDER> r;
    r.s = u.s;
#pragma unroll
    for (int k = ORDER == 1 ? 1 : 0; k <= ORDER; ++k) r.w[k] = limb_of(u.w[k]);
    return r;
}

// interpolation of one component of the fixed-point tile (extents SX, SY, lower halo H)
template <int ORDER, int DIM, int H>
__device__ __forceinline__ long long interp_q(const long long* __restrict__ F, int SX, int SY, const AxisQ<ORDER>& sx,
                                              const AxisQ<ORDER>& sy, const AxisQ<ORDER>& sz) {
    const long long* r = F + ((sz.s + H) * SY + (DIM == 3 ? sy.s + H : 0)) * SX + (sx.s + H);
    if constexpr (ORDER == 1) {
        if constexpr (DIM == 3) {
            const int SP = SX * SY;
            const long long a00 = lerpq(r[0], r[1], sx.w[1]), a10 = lerpq(r[SX], r[SX + 1], sx.w[1]);
            const long long a01 = lerpq(r[SP], r[SP + 1], sx.w[1]), a11 = lerpq(r[SP + SX], r[SP + SX + 1], sx.w[1]);
            return lerpq(lerpq(a00, a10, sy.w[1]), lerpq(a01, a11, sy.w[1]), sz.w[1]);
        } else {
            return lerpq(lerpq(r[0], r[1], sx.w[1]), lerpq(r[SX], r[SX + 1], sx.w[1]), sz.w[1]);
        }
    } else {
        AccQ vol;
#pragma unroll
        for (int c = 0; c <= ORDER; ++c) {
            AccQ pl;
#pragma unroll
            for (int b = 0; b <= (DIM == 3 ? ORDER : 0); ++b) {
                const long long* row = r + (c * SY + b) * SX;
                AccQ line;
#pragma unroll
                for (int a = 0; a <= ORDER; ++a) line.mac(row[a], sx.w[a]);
                if constexpr (DIM == 3) pl.mac(line.get(), sy.w[b]);
                else vol.mac(line.get(), sz.w[c]);
            }
            if constexpr (DIM == 3) vol.mac(pl.get(), sz.w[c]);
        }
        return vol.get();
    }
}

// ---- current amplitudes ----------------------------------------------------
// |value| = m 2^e with m < 2^63 and at least 58 significant bits; es = e << 20
// plus the sign in bit 31, modulo 2^32: products add it
struct Amp {
    u64 m;
    unsigned es;
};
__device__ __forceinline__ int exp_field(double x) {
    return (int)(((u64)__double_as_longlong(x) >> 52) & 0x7FFull);
}
__device__ __forceinline__ Amp amp_of(double x) {
    const u64 b = (u64)__double_as_longlong(x);
    const unsigned h = (unsigned)(b >> 32), lo = (unsigned)b;
    const unsigned mh = ((h & 0xFFFFFu) << 10) | (lo >> 22) | 0x40000000u;
    // zero and subnormals (below 2^-1022) are taken as zero
    return Amp{(h & 0x7FF00000u) == 0u ? 0ull : ((u64)mh << 32) | (lo << 10), (h & 0xFFF00000u) - (1085u << 20)};
}
__device__ __forceinline__ Amp amp_mul(const Amp& a, const Amp& b) {
    return Amp{mulhi(a.m, b.m), a.es + b.es + (64u << 20)};
}
// a times a Q62 number
__device__ __forceinline__ Amp amp_scale(const Amp& a, q62 p) {
    const u64 v = (u64)(p < 0 ? -p : p);
    unsigned h = (unsigned)(v >> 32), lo = (unsigned)v, es = a.es + (3u << 20) + ((unsigned)((u64)p >> 32) & 0x80000000u);
    if (h == 0u) {
        h = lo;
        lo = 0u;
        es -= 32u << 20;
    }
    const int l = __clz((int)h);
    const u64 n = ((u64)__funnelshift_l(lo, h, l) << 32) | (lo << (l & 31));
    return Amp{v == 0ull ? 0ull : mulhi(a.m, n >> 1), es - ((unsigned)l << 20)};
}
// A current contribution, amplitude x weight, rounded to nearest; false if there
// is none: a weight of zero, or a few units below it by the roundings of its
// factors.  Beside that rounding mulhi drops up to 2 units of 2^(e + 2): a
// current's amplitudes have m >= 2^58, so that is at most 2^-55 of the amplitude.
__device__ __forceinline__ bool contribution(const Amp& a, q62 T, double& v) {
    const u64 jm = mulhi(a.m, (u64)T);  // value jm 2^(e + 2)
    v = pack_double<true>(jm, a.es + (1087u << 20));
    return (int)(T >> 32) >= 0 && jm != 0ull;
}
// the exponent fields of a factor q w whose product with any of three
// prefactors, and every contribution of that, is a normal double (lo > hi: none)
struct ExpRange {
    int lo, hi;
};
__device__ __forceinline__ ExpRange exp_range(double a, double b, double c) {
    const int ea = exp_field(a), eb = exp_field(b), ec = exp_field(c);
    const int lo = min(ea, min(eb, ec)), hi = max(ea, max(eb, ec));
    if (lo == 0 || hi == 0x7FF) return ExpRange{1, 0};
    return ExpRange{max(1, 1246 - lo), min(0x7FE, 2846 - hi)};  // products within 2^-800 .. 2^800
}
__device__ __forceinline__ bool in_range(const ExpRange& r, int e) { return e >= r.lo && e <= r.hi; }

}  // namespace
