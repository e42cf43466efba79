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
//   vector real v = b 2^(E - o - 56), |b| < 2^56, b = b1 2^28 + b0 with both
//              limbs carrying v's sign; split in registers per hop. E is a
//              running block exponent per output site and rhs, o the exponent
//              of the hop's link block;
//   product    a b = a1 b1 2^56 + (a1 b0 + a0 b1) 2^28 + a0 b0: the first two
//              terms go to two 64-bit accumulators per output real (three
//              IMAD.WIDE a real product), a0 b0 is dropped.
//
// Bounds: an output real sums 96 products, so |S2| <= 96 2^55 and
// |S1| <= 96 (2^55 + 2^55) < 2^63. Against the largest product the dropped
// term is at most 2^-56, the vector rounding 2^-56, the link rounding 2^-56
// (reals within 4 of the block's largest are exact) and the final shift
// 2^-56; 96 FP64 fused multiply-adds round at 2^-53 of their running sum.
// Measured against quad-precision sums (Haar links, 8^4 and two ragged
// lattices): 1.2e-16 of the result for Gaussian vectors, 0.7e-16 for Z2 ones
// (1.7e-16 and 1.1e-16 at mu = 0.1); the FMA kernel 3.5e-16 for all of them.
//
// What bounds it: the register ports. An IMAD.WIDE with fresh operands (two
// factors, a 64-bit accumulator read and written) takes 3.3 to 4.2 cycles of
// a scheduler instead of 2; the 108 of a hop and rhs are 57 % of the time, the
// limb splitting 14 %, the rest link loads, addresses and the E test. One rhs
// a thread at 16 warps per SM is as fast as two at 12 (48^3x12, n = 8: 1.79 and
// 1.78 ms) or faster (32^3x8, n = 4: 178 us against 191); four need 255
// registers (8 warps a SM) and lose.
// Time per launch, FMA kernel -> this one: 48^3x12, n = 8: 5.24 -> 1.79 ms;
// 32^3x8, n = 8: 1055 -> 361 us; 24^3x6, n = 4: 305 -> 68 us; 16^4, n = 4: 156
// -> 52 us; 8^4, n = 1: 45 -> 8 us.
//
// E starts one above the first neighbour's largest exponent and grows when a
// later neighbour exceeds it; the accumulators are then shifted (rounded).
// Sites whose neighbours hold non-finite numbers, or only numbers outside
// 2^-900 .. 2^900, are recomputed with FP64 arithmetic (fx_site_fp64), so
// NaN, infinities and extreme ranges come out as from FP64 sums. Fields whose
// links differ in size by more than a factor of 16 inside a direction, or
// are not finite, keep the double storage and the FMA kernel.
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

// A stored real as double (exact for |l| >= 2^(e - 3)).
__device__ __forceinline__ double fx_link_real(int a1, int a0, int e) {
    const long long v = ((long long)a1 << 28) + a0;
    return (double)v * scalbn(1.0, e - 55);
}

// Limbs of v 2^(o - E + 56), negated for a backward hop; sh = E - o + 1030 -
// (exponent field of v) >= 8 low bits of the left-aligned mantissa go.
template <bool NEG>
__device__ __forceinline__ void fx_limbs(unsigned hi, unsigned lo, int k, int& b1, int& b0) {
    const int sh = k - (int)((hi << 1) >> 21);
    const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;
    const unsigned ml = lo << 11;
    unsigned long long u;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.u64 %0, t, %3;\n\t}" : "=l"(u) : "r"(ml), "r"(mh), "r"(sh));
    const unsigned ul = (unsigned)u, uh = (unsigned)(u >> 32);
    // the sign by a multiplication: the FMA pipe has room where the ALU has none
    const int s = (int)hi >> 31;
    const int sg = (NEG ? ~s : s) | 1;
    b0 = (int)(ul & 0x0fffffffu) * sg;
    b1 = (int)__funnelshift_r(ul, uh, 28) * sg;
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

// D in of one site and rhs in FP64 arithmetic (rare sites, see above).
template <int LAYOUT>
static __device__ __noinline__ void fx_site_fp64(const DslashArgs& a, int p, int h, int k, double2* out) {
    const Geom& g = a.g;
    const int vh = g.vh, q = 1 - p;
    const int xh = h % g.hx;
    int r = h / g.hx;
    const int y = r % g.L[1];
    r /= g.L[1];
    const int z = r % g.L[2], t = r / g.L[2];
    const int x = 2 * xh + ((p + y + z + t) & 1);
    double2 acc[3];
    for (int c = 0; c < 3; ++c) acc[c] = make_double2(0.0, 0.0);
    const double2* in = reinterpret_cast<const double2*>(a.in[k]) + (a.both ? (size_t)q * 3 * vh : 0);
#pragma unroll 1
    for (int e = a.t_only ? 12 : 0; e < 16; ++e) {
        const int mu = e >> 2, hop = e & 3, naik = hop >> 1, back = hop & 1;
        const int d = (naik ? 3 : 1) * (back ? -1 : 1);
        const int coord = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : t;
        const int stride = mu == 1 ? g.sy : mu == 2 ? g.sz : g.st;
        const int cn = wrap(coord + d, g.L[mu]);
        const int hn = mu == 0 ? h - xh + (cn >> 1) : h + (cn - coord) * stride;
        const int4* lk = reinterpret_cast<const int4*>(naik ? a.N : a.U) + (size_t)((back ? q : p) * 4 + mu) * 9 * vh +
                         (back ? hn : h);
        const int ex = a.fx_exp[naik * 4 + mu];
        const double f = (mu == 3 && a.has_mu) ? (hop == 0 ? a.ft1 : hop == 1 ? a.bt1 : hop == 2 ? a.ft3 : a.bt3) : 1.0;
        double2 v[3];
        for (int c = 0; c < 3; ++c) v[c] = in[spinor_index<LAYOUT>(hn, c, vh)];
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                const int4 w = lk[(size_t)(back ? 3 * j + i : 3 * i + j) * vh];
                const double2 m = make_double2(fx_link_real(w.x, w.y, ex) * f, fx_link_real(w.z, w.w, ex) * f);
                if (back)
                    cmsub_conj(acc[i], m, v[j]);
                else
                    cmadd(acc[i], m, v[j]);
            }
    }
    for (int c = 0; c < 3; ++c) out[c] = acc[c];
}

template <int R, int LAYOUT>
struct FxHops {
    const DslashArgs& a;
    const uint4* in[R];
    int vh, p, h, x, y, z, t;
    long long s2[R][6], s1[R][6];   // (re, im) of the three output colours
    int E[R];
    unsigned nz[R];
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
            nz[j] = 0u;
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
            const char* lk = reinterpret_cast<const char*>(NAIK ? a.N : a.U) + (size_t)((BACK ? 1 - p : p) * 4 + mu) * 9 * plane;
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
            nz[j] |= big;
            const int en = (int)(big >> 21) - 1022 + o;
            // the vote keeps the branch uniform: most hops skip it without the
            // divergence bookkeeping of a lane-wise branch (9 % of the kernel)
            if (__any_sync(__activemask(), en > E[j])) {
                if (en > E[j]) {
                    const int d = en + kFxHead - E[j];
                    E[j] = en + kFxHead;
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        s2[j][i] = fx_shift(s2[j][i], d);
                        s1[j][i] = fx_shift(s1[j][i], d);
                    }
                }
            }
            const int k = E[j] - o + 1030;
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
            nz[j] |= __shfl_xor_sync(0xffffffffu, nz[j], 8);
            nz[j] |= __shfl_xor_sync(0xffffffffu, nz[j], 16);
            const int d = em - E[j];
            E[j] = em;
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
        }
    }

    // whether rhs j left the range of the fixed-point sums
    __device__ __forceinline__ bool rare(int j) const {
        return E[j] > kFxCeil || (E[j] == kFxFloor && nz[j] != 0u) || a.fx_slow;
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
        if (SPLIT == 1 && v >= vh) continue;
        const int h = visit_site(v < vh ? v : vh - 1, a.g);
        FxHops<R, LAYOUT> hops(a, p, h, k0);
        if (SPLIT == 1) {
            hops.run(a.t_only ? 3 : 0, 4);
        } else {
            const int mu = lane >> 3;
            if (!a.t_only || mu == 3) hops.run(mu, mu + 1);
            hops.combine();
            if (mu != 0 || v >= vh) continue;
        }
        const bool neg = a.cd < 0.0;   // cd is +1 or -1 (checked by the launcher)
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = k0 + j;
            double2 w[3];
            if (hops.rare(j)) {
                fx_site_fp64<LAYOUT>(a, p, h, k, w);
                if (neg)
                    for (int c = 0; c < 3; ++c) w[c] = make_double2(-w[c].x, -w[c].y);
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) w[c] = make_double2(hops.value(j, 2 * c, neg), hops.value(j, 2 * c + 1, neg));
            }
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
    block_reduce_finish<R>(a, k0, red0, red1);
}

// Temporal factor f as a 55-bit mantissa in limbs and an exponent.
inline bool fx_factor(double f, int* f1, int* f0, int* fe) {
    if (!std::isfinite(f) || f == 0.0) return false;
    int e = 0;
    const double m = std::frexp(f, &e);
    const long long v = std::llrint(std::ldexp(m, 55));
    const long long lo = (long long)((unsigned long long)v << 36) >> 36;
    *f0 = (int)lo;
    *f1 = (int)((v - lo) >> 28);
    *fe = e;
    return e > -400 && e < 400;
}

template <int R, int SPLIT, int EPI, int LAYOUT, int MAXT, int MINB>
cudaError_t launch_fx64(const DslashArgs& args, cudaStream_t s) {
    const int G = args.nrhs / R;
    if (G < 1 || G * R != args.nrhs || G > 8) return cudaErrorInvalidValue;
    if (args.cd != 1.0 && args.cd != -1.0) return cudaErrorInvalidValue;
    if (args.both && args.red_mode != RED_NONE) return cudaErrorInvalidValue;
    DslashArgs a = args;
    a.fx_slow = 0;
    if (a.has_mu) {
        const double f[4] = {a.ft1, a.bt1, a.ft3, a.bt3};
        for (int i = 0; i < 4; ++i)
            if (!fx_factor(f[i], &a.fx_f1[i], &a.fx_f0[i], &a.fx_fe[i])) a.fx_slow = 1;
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
    const unsigned blocks = plan_tiles(a, ((long long)a.g.vh + spb - 1) / spb);
    kern<<<dim3(blocks, a.both ? 2 : 1), dim3(bx, G), 0, s>>>(a);
    return finish_launch(a, blocks, s);
}

}  // namespace hisq
