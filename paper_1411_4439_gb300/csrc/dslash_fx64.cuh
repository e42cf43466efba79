// FP64 multi-rhs Dslash (Eq. 3 on a bundle, Eq. 4) on the integer pipes.
//
// The FP64 pipe of this GPU retires 2 fused multiply-adds a clock and SM, the
// 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE) 60 (both measured), and
// the FMA kernel ran at 98 % of the FP64 pipe. This kernel forms the same
// sums in block fixed point, exactly but for the roundings listed below:
//
//   link real  l = a 2^(e - 55), e the exponent of the (field, direction)
//              block (every |l| < 2^e), a = a1 2^28 + a0 with |a1| <= 2^27 and
//              |a0| <= 2^27; packed once when the field is loaded;
//   vector real v = b 2^(E - o - 56), |b| <= 2^56, b = b1 2^28 + b0 with |b1| <= 2^28
//              and |b0| <= 2^27; split in registers per hop. E is a running
//              block exponent per output site and rhs, o the exponent of the
//              hop's link block;
//   product    a b = a1 b1 2^56 + (a1 b0 + a0 b1) 2^28 + a0 b0: the first two
//              terms go to two 64-bit accumulators per output real (three
//              IMAD.WIDE a real product), a0 b0 is dropped.
//
// Bounds: an output real sums 96 products, so |S2| <= 96 2^55 and
// |S1| <= 96 (2^54 + 2^55) < 2^63. In units of 2^E a product loses at most 2^-56
// to the link's rounding, 2^-57 to the vector's and 2^-57 to the dropped term,
// so a sum is off by at most 25 x 2^(E - 53), 0.35 x 2^(E - 53) in the root mean
// square for Haar links. 2^E is 2 to 4 times the largest neighbour real times
// the block scale 2^o, so it says nothing about one output: the link may be zero
// or small where the neighbour is large, or lead to another colour. What an FP64
// sum loses follows its own partial sums, and so does the test here: an output
// real counts only if its sum, looked at after every hop, came to 2^(E - 6) at
// least once (kFxReach); the sites of other outputs are formed again by fx_redo
// with FP64 multiply-adds on the double links, which the field keeps beside the
// fixed-point ones. Root mean square errors (8000 to 40000 sites in numpy
// integers against long double):
//
//                                             this kernel   FP64 multiply-adds
//   site norm: Haar links x 0.9                  0.9e-16          3.7e-16
//              Haar links x 0.51                 1.3e-16          3.7e-16
//   real against the sum of its |products|:
//              Haar links                        1.6e-17          7.1e-17
//              a single neighbour                5.2e-17          5.2e-17
//              a single neighbour and colour     1.2e-16          0.5e-16
//              one colour 1/16 of the others,
//              links diagonal                    2.0e-16          0.7e-16
//
// and no real is off by more than 1600 units of 2^-53 of the sum of its
// |products| (multiply-adds: 96). Links that are mostly diagonal, real or
// otherwise thin, where a vector's parts stay apart, keep to multiply-adds (see
// plan_links). Rounding the vectors and balancing their low limb halves the error
// for 2.5 % of the time; the looks at the sums take 1.5 %. At a limit of 2^(E - 5)
// Gaussian vectors at mu = 0.1 have a thousandth of the sites formed again, 3 to 8 %
// of the time (8^4, n = 1: 12.7 us against 8.4); at 2^(E - 6) it does not show.
//
// What bounds it: the register ports. An IMAD.WIDE with fresh operands (two
// factors, a 64-bit accumulator read and written) takes 3.3 to 4.2 cycles of
// a scheduler instead of 2; the 108 of a hop and rhs are 57 % of the time, the
// limb splitting 14 %, the rest link loads, addresses and the E test. One rhs
// a thread at 16 warps per SM is as fast as two at 12 (48^3x12, n = 8, before the
// looks at the sums: 1.79 and 1.78 ms) or faster (32^3x8, n = 4: 178 us against
// 191); four need 255 registers (8 warps a SM) and lose.
// Time per launch, FMA kernel -> this one: 48^3x12, n = 8: 5.24 -> 1.87 ms;
// 32^3x8, n = 8: 1055 -> 376 us; 24^3x6, n = 4: 305 -> 67 us; 16^4, n = 4: 156
// -> 52 us; 8^4, n = 1: 45 -> 8 us.
//
// E starts one above the first neighbour's largest exponent and grows when a
// later neighbour exceeds it; the accumulators are then shifted (rounded).
// Sites with a neighbour that is not finite or beyond 2^900 go through fx_redo
// too, so NaN, infinities and extreme ranges come out as from FP64 sums.
//
// Full-lattice operators take both parities in one launch (a.both): 24^3x6, n =
// 4, M^dag 163 -> 143 us, the waves of the second parity fill the first's tail.
//
// A thread takes one output site and R rhs; with SPLIT = 4 the four lanes of
// a site take one direction each and add their accumulators with shuffles
// (lattices too small to fill the SMs).
#pragma once

#include "dslash_impl.cuh"

namespace hisq {

constexpr int kFxFloor = -900;   // lowest block exponent
constexpr int kFxCeil = 900;     // above: FP64 path
constexpr int kFxHead = 1;       // bits a new block exponent leaves above its vector
constexpr int kFxReach = 6;      // a sum that never came within 2^-kFxReach of 2^E is formed in FP64

// Limbs of v 2^(o - E + 56) rounded, negated for a backward hop; sh = E - o +
// 1029 - (exponent field of v) >= 7 low bits of the left-aligned mantissa go,
// one bit stays below the unit for the rounding.
template <bool NEG>
__device__ __forceinline__ void fx_limbs(unsigned hi, unsigned lo, int k, int& b1, int& b0) {
    const int sh = k - (int)((hi << 1) >> 21);
    const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;
    const unsigned ml = lo << 11;
    unsigned long long u;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.u64 %0, t, %3;\n\t}" : "=l"(u) : "r"(ml), "r"(mh), "r"(sh));
    // + 1 rounds, + 2^28 (2^27 units) makes the low limb -2^27 .. 2^27 - 1
    u += (1ull << 28) + 1;
    const unsigned ul = (unsigned)u, uh = (unsigned)(u >> 32);
    // the sign by a multiplication: the FMA pipe has room where the ALU has none
    const int s = (int)hi >> 31;
    const int sg = (NEG ? ~s : s) | 1;
    b0 = ((int)((ul >> 1) & 0x0fffffffu) - (1 << 27)) * sg;
    b1 = (int)__funnelshift_r(ul, uh, 29) * sg;
}

__device__ __forceinline__ void fx_mac(long long& s, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
}

// s / 2^d rounded to nearest, d >= 1.
__device__ __forceinline__ long long fx_shift(long long s, int d) {
    d = d > 63 ? 63 : d;
    return (s + (1ll << (d - 1))) >> d;
}

// Factor f of a temporal hop as fm 2^fe, fm 2^55 in limbs.
__device__ __forceinline__ void fx_scale(int& x1, int& x0, int f1, int f0) {
    long long cross = 0, top = 0;
    fx_mac(cross, x1, f0);
    fx_mac(cross, x0, f1);
    fx_mac(top, x1, f1);
    const long long v = 2 * top + ((cross + (1ll << 26)) >> 27);   // (x f) / 2^55
    x0 = (int)((unsigned)v << 4) >> 4;
    x1 = (int)((v - x0) >> 28);
}

// D in of the sites (h of the lanes in mask) and rhs k in FP64 arithmetic on the
// double links; every lane of the warp calls it and the lanes in mask get w.
// Two sites a pass, a lane per hop: one flagged site costs the FP64 pipe a
// sixteenth of what it costs a lane on its own.
template <int LAYOUT>
static __device__ __noinline__ void fx_redo(const DslashArgs& a, int p, int k, unsigned mask, int h, double2 (&w)[3]) {
    const Geom& g = a.g;
    const int vh = g.vh, q = 1 - p, lane = threadIdx.x & 31;
    const int mu = (lane & 15) >> 2, hop = lane & 3, naik = hop >> 1, back = hop & 1;
    const int d = (naik ? 3 : 1) * (back ? -1 : 1);
    const double f = (mu == 3 && a.has_mu) ? (hop == 0 ? a.ft1 : hop == 1 ? a.bt1 : hop == 2 ? a.ft3 : a.bt3) : 1.0;
    const double2* in = reinterpret_cast<const double2*>(a.in[k]) + (a.both ? (size_t)q * 3 * vh : 0);
    const double2* block = reinterpret_cast<const double2*>(naik ? a.N : a.U) + (size_t)((back ? q : p) * 4 + mu) * 9 * vh;
#pragma unroll 1
    while (mask) {
        const int first = __ffs(mask) - 1;
        mask &= mask - 1;
        const int second = mask ? __ffs(mask) - 1 : first;
        mask &= mask - 1;
        const int hs = __shfl_sync(0xffffffffu, h, lane < 16 ? first : second);
        double2 acc[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] = make_double2(0.0, 0.0);
        if (mu == 3 || !a.t_only) {
            const int xh = hs % g.hx;
            int r = hs / g.hx;
            const int y = r % g.L[1];
            r /= g.L[1];
            const int z = r % g.L[2], t = r / g.L[2];
            const int x = 2 * xh + ((p + y + z + t) & 1);
            const int coord = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : t;
            const int stride = mu == 1 ? g.sy : mu == 2 ? g.sz : g.st;
            const int cn = wrap(coord + d, g.L[mu]);
            const int hn = mu == 0 ? hs - xh + (cn >> 1) : hs + (cn - coord) * stride;
            const double2* lk = block + (back ? hn : hs);
            double2 v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = __ldg(in + spinor_index<LAYOUT>(hn, c, vh));
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const double2 l = __ldg(lk + (size_t)(back ? 3 * j + i : 3 * i + j) * vh);
                    const double2 m = make_double2(l.x * f, l.y * f);
                    if (back)
                        cmsub_conj(acc[i], m, v[j]);
                    else
                        cmadd(acc[i], m, v[j]);
                }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, o);
                acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, o);
            }
            const int from = lane == first ? 0 : 16;
            const double re = __shfl_sync(0xffffffffu, acc[c].x, from), im = __shfl_sync(0xffffffffu, acc[c].y, from);
            if (lane == first || lane == second) w[c] = make_double2(re, im);
        }
    }
}

// The upper halves of two 32-bit words, each with the bits of its sign flipped
// away: |word| / 2^16 (rounded down for negative words) side by side.
__device__ __forceinline__ unsigned fx_tops(unsigned a, unsigned b) {
    unsigned v, s;
    asm("prmt.b32 %0, %1, %2, 0x7632;" : "=r"(v) : "r"(a), "r"(b));
    asm("prmt.b32 %0, %1, %2, 0xffbb;" : "=r"(s) : "r"(a), "r"(b));   // sign bytes
    return v ^ s;
}

// Two halves of 16 bits shifted right by d >= 0.
__device__ __forceinline__ unsigned fx_shift_tops(unsigned t, int d) {
    return d > 15 ? 0u : (t >> d) & ((0xffffu >> d) * 0x10001u);
}

template <int R, int LAYOUT>
struct FxHops {
    const DslashArgs& a;
    const uint4* in[R];
    int vh, p, h, x, y, z, t;
    long long s2[R][6], s1[R][6];   // (re, im) of the three output colours
    int E[R];
    unsigned peak[R];               // largest exponent field of a neighbour real, at bit 21
    unsigned tops[R][3];            // per colour (re, im): OR over the hops of the sum's size, 2^(E - 7) a unit
    uint4 cur[R][3];                // the next hop's neighbour vectors, as loaded
    // the direction at hand: coordinate, extent, half-index step (0 shift but x)
    int mu, c, ext, stride, half;

    __device__ __forceinline__ FxHops(const DslashArgs& args, int p_, int h_, int k0) : a(args) {
        vh = a.g.vh;
        p = p_;
        h = h_;
        const int xh = h % a.g.hx;
        int r = h / a.g.hx;
        y = r % a.g.L[1];
        r /= a.g.L[1];
        z = r % a.g.L[2];
        t = r / a.g.L[2];
        x = 2 * xh + ((p + y + z + t) & 1);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            in[j] = reinterpret_cast<const uint4*>(a.in[k0 + j]) + (a.both ? (size_t)(1 - p) * 3 * vh : 0);
            E[j] = kFxFloor;
            peak[j] = 0u;
#pragma unroll
            for (int c = 0; c < 3; ++c) tops[j][c] = 0u;
#pragma unroll
            for (int c = 0; c < 6; ++c) s2[j][c] = s1[j][c] = 0ll;
        }
    }

    __device__ __forceinline__ void set_direction(int m) {
        mu = m;
        c = m == 0 ? x : m == 1 ? y : m == 2 ? z : t;
        ext = m == 0 ? a.g.L[0] : m == 1 ? a.g.L[1] : m == 2 ? a.g.L[2] : a.g.L[3];
        stride = m == 0 ? 1 : m == 1 ? a.g.sy : m == 2 ? a.g.sz : a.g.st;
        half = m == 0 ? 1 : 0;
    }

    // neighbour of hop HOP (+1, -1, +3, -3) of the direction at hand
    template <int HOP>
    __device__ __forceinline__ int neighbour() const {
        int cn;
        if (HOP & 1) {
            cn = c - (HOP == 1 ? 1 : 3);
            cn += cn < 0 ? ext : 0;
        } else {
            cn = c + (HOP == 0 ? 1 : 3);
            cn -= cn >= ext ? ext : 0;
        }
        return h + ((cn >> half) - (c >> half)) * stride;
    }

    template <int HOP>
    __device__ __forceinline__ void issue() {
        const int hn = neighbour<HOP>();
#pragma unroll
        for (int j = 0; j < R; ++j) {
#pragma unroll
            for (int i = 0; i < 3; ++i) cur[j][i] = __ldg(in[j] + spinor_index<LAYOUT>(hn, i, vh));
        }
    }

    // one hop; the vectors of the next one (of direction `after` for the last
    // hop, none if it is negative) are loaded while this one is multiplied
    template <int HOP>
    __device__ __forceinline__ void hop(int after) {
        constexpr bool BACK = HOP & 1;
        constexpr int NAIK = HOP >> 1;
        int4 m[9];
        {
            const size_t plane = (size_t)vh * sizeof(int4);
            const char* lk = reinterpret_cast<const char*>(NAIK ? a.N_fx : a.U_fx) + (size_t)((BACK ? 1 - p : p) * 4 + mu) * 9 * plane;
            const unsigned off = (unsigned)(BACK ? neighbour<HOP>() : h) * (unsigned)sizeof(int4);
#pragma unroll
            for (int e = 0; e < 9; ++e) m[e] = __ldcs(reinterpret_cast<const int4*>(lk + e * plane + off));
        }
        int o = a.fx_exp[NAIK * 4 + mu];
        const bool scaled = mu == 3 && a.has_mu;
        if (scaled) o += a.fx_fe[HOP];
        int v1[R][6], v0[R][6];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            unsigned big = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) big = max(big, max(cur[j][i].y << 1, cur[j][i].w << 1));
            peak[j] = max(peak[j], big);
            const int en = (int)(big >> 21) - 1022 + o;
            // the vote keeps the branch uniform: most hops skip it without the
            // divergence bookkeeping of a lane-wise branch (9 % of the kernel)
            if (__any_sync(__activemask(), en > E[j])) {
                if (en > E[j]) {
                    const int d = en + kFxHead - E[j];
                    E[j] = en + kFxHead;
#pragma unroll
                    for (int i = 0; i < 3; ++i) tops[j][i] = fx_shift_tops(tops[j][i], d);
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        s2[j][i] = fx_shift(s2[j][i], d);
                        s1[j][i] = fx_shift(s1[j][i], d);
                    }
                }
            }
            const int k = E[j] - o + 1029;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                fx_limbs<BACK>(cur[j][i].y, cur[j][i].x, k, v1[j][2 * i], v0[j][2 * i]);
                fx_limbs<BACK>(cur[j][i].w, cur[j][i].z, k, v1[j][2 * i + 1], v0[j][2 * i + 1]);
            }
        }
        if constexpr (HOP < 3) {
            issue<HOP + 1>();
        } else if (after >= 0) {
            set_direction(after);
            issue<0>();
        }
        if (scaled) {
            const int f1 = a.fx_f1[HOP], f0 = a.fx_f0[HOP];
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                fx_scale(m[e].x, m[e].y, f1, f0);
                fx_scale(m[e].z, m[e].w, f1, f0);
            }
        }
        // forward m_ic v_c, backward conj(m_ci) (-v_c): the negated part of v
        // is Im v forward (re -= Im m Im v), Re v backward (im -= Im m Re v)
#pragma unroll
        for (int col = 0; col < 3; ++col) {
            int n1[R], n0[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                n1[j] = -v1[j][2 * col + (BACK ? 0 : 1)];
                n0[j] = -v0[j][2 * col + (BACK ? 0 : 1)];
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int4 e = m[BACK ? 3 * col + i : 3 * i + col];
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    const int r1 = v1[j][2 * col], r0 = v0[j][2 * col], w1 = v1[j][2 * col + 1], w0 = v0[j][2 * col + 1];
                    const int x1 = BACK ? w1 : n1[j], x0 = BACK ? w0 : n0[j];   // Im m factor of re
                    const int y1 = BACK ? n1[j] : r1, y0 = BACK ? n0[j] : r0;   // Im m factor of im
                    fx_mac(s2[j][2 * i], e.x, r1);
                    fx_mac(s1[j][2 * i], e.x, r0);
                    fx_mac(s2[j][2 * i + 1], e.x, w1);
                    fx_mac(s1[j][2 * i + 1], e.x, w0);
                    fx_mac(s2[j][2 * i], e.z, x1);
                    fx_mac(s1[j][2 * i], e.y, r1);
                    fx_mac(s2[j][2 * i + 1], e.z, y1);
                    fx_mac(s1[j][2 * i + 1], e.y, w1);
                    fx_mac(s1[j][2 * i], e.z, x0);
                    fx_mac(s1[j][2 * i + 1], e.z, y0);
                    fx_mac(s1[j][2 * i], e.w, x1);
                    fx_mac(s1[j][2 * i + 1], e.w, y1);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < R; ++j) note_sizes(j);
    }

    __device__ __forceinline__ void note_sizes(int j) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
            tops[j][i] |= fx_tops((unsigned)(s2[j][2 * i] >> 32), (unsigned)(s2[j][2 * i + 1] >> 32));
    }

    // the hops of the directions [first, last)
    __device__ __forceinline__ void run(int first, int last) {
        set_direction(first);
        issue<0>();
#pragma unroll 1
        for (int m = first; m < last; ++m) {
            hop<0>(-1);
            hop<1>(-1);
            hop<2>(-1);
            hop<3>(m + 1 < last ? m + 1 : -1);
        }
    }

    // sum over the four lanes (8 apart) that hold a site's directions
    __device__ __forceinline__ void combine() {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            int em = max(E[j], __shfl_xor_sync(0xffffffffu, E[j], 8));
            em = max(em, __shfl_xor_sync(0xffffffffu, em, 16));
            peak[j] = max(peak[j], __shfl_xor_sync(0xffffffffu, peak[j], 8));
            peak[j] = max(peak[j], __shfl_xor_sync(0xffffffffu, peak[j], 16));
            const int d = em - E[j];
            E[j] = em;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                tops[j][i] = fx_shift_tops(tops[j][i], d);
                tops[j][i] |= __shfl_xor_sync(0xffffffffu, tops[j][i], 8);
                tops[j][i] |= __shfl_xor_sync(0xffffffffu, tops[j][i], 16);
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                long long u = s2[j][c], w = s1[j][c];
                if (d > 0) {
                    u = fx_shift(u, d);
                    w = fx_shift(w, d);
                }
                u += __shfl_xor_sync(0xffffffffu, u, 8);
                w += __shfl_xor_sync(0xffffffffu, w, 8);
                u += __shfl_xor_sync(0xffffffffu, u, 16);
                w += __shfl_xor_sync(0xffffffffu, w, 16);
                s2[j][c] = u;
                s1[j][c] = w;
            }
            note_sizes(j);
        }
    }

    // Whether rhs j needs FP64 arithmetic: a neighbour that is not finite or too
    // large, or an output real whose sums stayed below 2^(E - kFxReach). (Neighbours
    // that are all zero give exact zeros.)
    __device__ __forceinline__ bool rare(int j) const {
        constexpr unsigned kSmall = (1u << (23 - kFxReach - 16)) - 1;   // hi word of 2^(E - kFxReach) is 2^(23 - kFxReach)
        bool low = false;
#pragma unroll
        for (int i = 0; i < 3; ++i) low = low || (tops[j][i] & 0xffffu) <= kSmall || (tops[j][i] >> 16) <= kSmall;
        return peak[j] >= 0xffe00000u || E[j] > kFxCeil || (low && peak[j] != 0u);
    }

    // (S2 2^28 + S1) 2^(E - 83), times sgn = +-1
    __device__ __forceinline__ double value(int j, int c, bool neg) const {
        long long v = s2[j][c] + ((s1[j][c] + (1ll << 27)) >> 28);
        v = neg ? -v : v;
        const double w = (double)v;
        return v == 0 ? 0.0 : __hiloint2double(__double2hiint(w) + ((E[j] - 55) << 20), __double2loint(w));
    }
};

template <int R, int SPLIT, int EPI, int LAYOUT, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) dslash_fx64_kernel(const __grid_constant__ DslashArgs a) {
    static_assert(SPLIT == 1 || SPLIT == 4, "a site takes one lane or one lane per direction");
    const int vh = a.g.vh;
    const int p = a.both ? (int)blockIdx.y : a.parity;
    const size_t half = a.both ? (size_t)p * 3 * vh : 0;   // of the output parity
    const int k0 = threadIdx.y * R;
    const int lane = threadIdx.x & 31;
    const int slot = SPLIT == 1 ? (int)threadIdx.x : (int)(threadIdx.x >> 5) * 8 + (lane & 7);
    const int spb = blockDim.x / SPLIT;
    double red0[R], red1[R];   // red1: largest |w|^2 until the loop ends
#pragma unroll
    for (int j = 0; j < R; ++j) red0[j] = red1[j] = 0.0;

    const int v0 = blockIdx.x * a.run * spb;
    for (int it = 0, v = v0 + slot; it < a.run && v - slot < vh; ++it, v += spb) {
        const int h = visit_site(v < vh ? v : vh - 1, a.g);
        FxHops<R, LAYOUT> hops(a, p, h, k0);
        bool mine = v < vh;
        if (SPLIT == 1) {
            hops.run(a.t_only ? 3 : 0, 4);
        } else {
            const int mu = lane >> 3;
            if (!a.t_only || mu == 3) hops.run(mu, mu + 1);
            hops.combine();
            mine = mine && mu == 0;
        }
        const bool neg = a.cd < 0.0;   // cd is +1 or -1 (checked by the launcher)
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = k0 + j;
            double2 w[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) w[c] = make_double2(hops.value(j, 2 * c, neg), hops.value(j, 2 * c + 1, neg));
            const bool again = mine && hops.rare(j);
            const unsigned mask = __ballot_sync(0xffffffffu, again);
            if (mask) {
                double2 u[3];
                fx_redo<LAYOUT>(a, p, k, mask, h, u);
                if (again) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) w[c] = neg ? make_double2(-u[c].x, -u[c].y) : u[c];
                }
            }
            if (!mine) continue;
            double2* o = reinterpret_cast<double2*>(a.out[k]) + half;
            double n2max = 0.0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const size_t i = spinor_index<LAYOUT>(h, c, vh);
                if constexpr (EPI != EPI_NONE) {
                    const double2 xv = __ldg(reinterpret_cast<const double2*>(a.x[k]) + half + i);
                    w[c].x = fma(a.cx, xv.x, w[c].x);
                    w[c].y = fma(a.cx, xv.y, w[c].y);
                    if constexpr (EPI == EPI_XY) {
                        const double2 yv = __ldg(reinterpret_cast<const double2*>(a.y[k]) + half + i);
                        w[c].x += yv.x;
                        w[c].y += yv.y;
                    }
                    if (a.red_mode == RED_DOT_XW) red0[j] = fma(xv.x, w[c].x, fma(xv.y, w[c].y, red0[j]));
                }
                o[i] = w[c];
                if (a.red_mode == RED_NORM_MAX_W) {
                    const double n2 = fma(w[c].x, w[c].x, w[c].y * w[c].y);
                    red0[j] += n2;
                    n2max = fmax(n2max, n2);
                }
            }
            red1[j] = fmax(red1[j], n2max);
        }
    }
    if (a.red_mode == RED_NONE) return;
    if (a.red_mode == RED_NORM_MAX_W) {
#pragma unroll
        for (int j = 0; j < R; ++j) red1[j] = sqrt(red1[j]);
    }
    __shared__ RedParts parts;
    tile_reduce<R>(a, k0, red0, red1, parts, true);
    block_finish<false>(a, parts);
}

// Temporal factor f (in fx64_usable's range) as a 55-bit mantissa in limbs and an exponent.
inline void fx_factor(double f, int* f1, int* f0, int* fe) {
    int e = 0;
    const double m = std::frexp(f, &e);
    const long long v = std::llrint(std::ldexp(m, 55));
    const long long lo = (long long)((unsigned long long)v << 36) >> 36;
    *f0 = (int)lo;
    *f1 = (int)((v - lo) >> 28);
    *fe = e;
}

template <int R, int SPLIT, int EPI, int LAYOUT, int MAXT, int MINB>
cudaError_t launch_fx64(const DslashArgs& args, cudaStream_t s) {
    const int G = args.nrhs / R;
    if (G < 1 || G * R != args.nrhs || G > 8) return cudaErrorInvalidValue;
    if (args.cd != 1.0 && args.cd != -1.0) return cudaErrorInvalidValue;
    if (args.both && args.red_mode != RED_NONE) return cudaErrorInvalidValue;
    if (!fx64_usable(args)) return cudaErrorInvalidValue;
    DslashArgs a = args;
    if (a.has_mu) {
        const double f[4] = {a.ft1, a.bt1, a.ft3, a.bt3};
        for (int i = 0; i < 4; ++i) fx_factor(f[i], &a.fx_f1[i], &a.fx_f0[i], &a.fx_fe[i]);
    }
    int bx = 128 / G;
    bx &= ~31;
    if (bx < 32) bx = 32;
    if (bx * G > MAXT) return cudaErrorInvalidValue;
    auto* kern = dslash_fx64_kernel<R, SPLIT, EPI, LAYOUT, MAXT, MINB>;
    static OccCache cache;
    int occ = 0;
    cudaError_t e = cached_occupancy(cache, kern, bx * G, 0, G, &occ);
    if (e != cudaSuccess) return e;
    const int spb = bx / SPLIT;
    const unsigned blocks = plan_tiles<false>(a, ((long long)a.g.vh + spb - 1) / spb);
    kern<<<dim3(blocks, a.both ? 2 : 1), dim3(bx, G), 0, s>>>(a);
    return finish_launch(a, blocks, s);
}

}  // namespace hisq
