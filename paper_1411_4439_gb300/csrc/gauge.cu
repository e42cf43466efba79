// Link packing and reconstruction (Sec. 1: links stored in fewer reals).
//
// Canonical input: complex128 [4][V][3][3], lexicographic site order.
// Internal output: per (parity, mu) block the stored components of V_h
// sites in the storage precision (FP64, FP32, or 16-bit fixed point with one
// scale per stored component): FP64 as [component][V_h]; FP32 and 16-bit as
// [component pair][V_h] (two components of a site in one 16- or 8-byte word)
// and the odd last component as [V_h] (link_offset). A warp's 32 consecutive
// sites read each word with one coalesced access.
//   R18: 9 components; R14: rows 1-2 and z with row3 = z conj(row1 x row2);
//   R12: rows 1-2 with row3 = (sigma/s) conj(row1 x row2).
// Every packed link is reconstructed here in FP64 and compared with the
// input; the largest deviation is returned so the loader can reject links
// that the chosen compression cannot represent.
#include "hisq_internal.cuh"

namespace hisq {

namespace {

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zsub(double2 a, double2 b) {
    return make_double2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double zabs(double2 a) { return sqrt(a.x * a.x + a.y * a.y); }

// conj(a x b) for rows a = m[0..2], b = m[3..5]
__device__ __forceinline__ void cross_conj(const double2* m, double2* c) {
    c[0] = zconj(zsub(zmul(m[1], m[5]), zmul(m[2], m[4])));
    c[1] = zconj(zsub(zmul(m[2], m[3]), zmul(m[0], m[5])));
    c[2] = zconj(zsub(zmul(m[0], m[4]), zmul(m[1], m[3])));
}

struct Site {
    int x, y, z, t, parity, h;
};

__device__ __forceinline__ Site site_of(const Geom& g, unsigned i) {   // i < V <= 2^27
    Site s;
    unsigned r = i;
    s.x = (int)(r % (unsigned)g.L[0]);
    r /= (unsigned)g.L[0];
    s.y = (int)(r % (unsigned)g.L[1]);
    r /= (unsigned)g.L[1];
    s.z = (int)(r % (unsigned)g.L[2]);
    s.t = (int)(r / (unsigned)g.L[2]);
    s.parity = (s.x + s.y + s.z + s.t) & 1;
    s.h = (int)(i >> 1);
    return s;
}

// staggered sign eta_mu(x) * bc(x, mu) of the link x -> x + hop mu (antiperiodic t)
__device__ __forceinline__ int staggered_sign(const Geom& g, const Site& s, int mu, int hop) {
    int e = 0;
    if (mu >= 1) e += s.x;
    if (mu >= 2) e += s.y;
    if (mu >= 3) e += s.z;
    int sg = (e & 1) ? -1 : 1;
    if (mu == 3 && s.t + hop >= g.L[3]) sg = -sg;
    return sg;
}

// Compute the `ncomp` stored complex numbers of one link and its reconstruct error.
__device__ __forceinline__ double encode(const double2* m, int recon, int sign, double inv_s,
                                         double2* enc) {
#pragma unroll
    for (int c = 0; c < 6; ++c) enc[c] = m[c];
    double err = 0.0;
    if (recon == 18) {
        enc[6] = m[6];
        enc[7] = m[7];
        enc[8] = m[8];
        return 0.0;
    }
    double2 cc[3];
    cross_conj(m, cc);
    double2 f;
    if (recon == 14) {
        int k = 0;
        double best = zabs(cc[0]);
        if (zabs(cc[1]) > best) { k = 1; best = zabs(cc[1]); }
        if (zabs(cc[2]) > best) { k = 2; best = zabs(cc[2]); }
        if (best > 0.0) {
            // z = row3_k / cc_k
            const double d = cc[k].x * cc[k].x + cc[k].y * cc[k].y;
            f = make_double2((m[6 + k].x * cc[k].x + m[6 + k].y * cc[k].y) / d,
                             (m[6 + k].y * cc[k].x - m[6 + k].x * cc[k].y) / d);
        } else {
            f = make_double2(0.0, 0.0);
        }
        enc[6] = f;
    } else {
        f = make_double2(sign > 0 ? inv_s : -inv_s, 0.0);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double2 r3 = zmul(f, cc[c]);
        err = fmax(err, zabs(zsub(r3, m[6 + c])));
    }
    return err;
}

__device__ __forceinline__ void atomic_max_nonneg(unsigned long long* bits, double v) {
    if (!(v >= 0.0)) v = __longlong_as_double(0x7ff0000000000000ll);   // NaN -> +inf
    atomicMax(bits, (unsigned long long)__double_as_longlong(v));
}

// bits of |v|: as unsigned integers they order like the values (NaN above
// infinity), and the ALU compares them 30 times faster than the FP64 pipe
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
__device__ __forceinline__ unsigned long long skip_nan(unsigned long long b) { return b > kInfBits ? 0ull : b; }
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}

// Stored component 6 of an R14 link (z = row3_k / conj(row1 x row2)_k for the
// largest k) or the factor of row 3 of an R12 one, and the largest deviation
// of row 3 = f conj(row1 x row2) from the input.
template <int RECON>
__device__ __forceinline__ double2 third_factor(const double2* m, int sign, double inv_s, double& err) {
    double2 cc[3];
    cross_conj(m, cc);
    double2 f;
    if (RECON == 14) {
        double n2[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) n2[c] = cc[c].x * cc[c].x + cc[c].y * cc[c].y;
        double2 ck = cc[0], mk = m[6];
        double d = n2[0];
        if (n2[1] > d) { ck = cc[1]; mk = m[7]; d = n2[1]; }
        if (n2[2] > d) { ck = cc[2]; mk = m[8]; d = n2[2]; }
        f = make_double2(0.0, 0.0);
        if (d > 0.0) {
            const double inv = 1.0 / d;
            f = make_double2((mk.x * ck.x + mk.y * ck.y) * inv, (mk.y * ck.x - mk.x * ck.y) * inv);
        }
    } else {
        f = make_double2(sign > 0 ? inv_s : -inv_s, 0.0);
    }
    double e2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double2 dv = zsub(zmul(f, cc[c]), m[6 + c]);
        e2 = fmax(e2, dv.x * dv.x + dv.y * dv.y);
    }
    err = fmax(err, sqrt(e2));
    return f;
}

// One pass over a field before it is packed; blockIdx.y = mu. Every block
// reduces its maxima in shared memory and issues one atomic per value; with
// atomics from every thread the pass took 5.6 to 6.9 ms at 48^3x12, now
// 0.19 ms (R18, 4.0 TB/s) and 1.08 ms (R14: FP64 pipe, 78 operations a link
// for the reconstruct check).
template <int RECON>
__global__ void __launch_bounds__(256) scan_kernel(Geom g, const double2* __restrict__ canon, int hop, double inv_s,
                                                   LinkScan* out) {
    constexpr int NC = RECON / 2;
    const unsigned V = 2u * (unsigned)g.vh;
    const int mu = blockIdx.y;
    unsigned long long mx[NC], hi = 0ull, lo = ~0ull;
    unsigned links = 0, thin = 0;
    double err = 0.0;
#pragma unroll
    for (int c = 0; c < NC; ++c) mx[c] = 0ull;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
        const double2* src = canon + ((size_t)mu * V + i) * 9;
        double2 m[9];
        unsigned long long link = 0ull;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            m[c] = src[c];
            link = umax64(link, umax64(abs_bits(m[c].x), abs_bits(m[c].y)));
        }
        // a NaN is its own link's matter: the scales of the others come from the numbers
        const bool nan = link > kInfBits;
#pragma unroll
        for (int c = 0; c < NC && (c < 6 || RECON == 18); ++c) {
            unsigned long long x = abs_bits(m[c].x), y = abs_bits(m[c].y);
            if (nan) {
                x = skip_nan(x);
                y = skip_nan(y);
            }
            mx[c] = umax64(mx[c], umax64(x, y));
        }
        hi = umax64(hi, link);
        if (link != 0ull) {
            lo = link < lo ? link : lo;
            ++links;
            // reals below 1/16 of the link's largest (four off its exponent)
            const long long small = (long long)link - (4ll << 52);
#pragma unroll
            for (int c = 0; c < 9; ++c)
                thin += ((long long)abs_bits(m[c].x) < small) + ((long long)abs_bits(m[c].y) < small);
        }
        if (RECON != 18) {
            const int sg = RECON == 12 ? staggered_sign(g, site_of(g, i), mu, hop) : 1;
            const double2 f = third_factor<RECON>(m, sg, inv_s, err);
            if (RECON == 14) mx[NC - 1] = umax64(mx[NC - 1], umax64(skip_nan(abs_bits(f.x)), skip_nan(abs_bits(f.y))));
        }
    }
    __shared__ unsigned long long s_v[12][8];
    unsigned long long v[12];
#pragma unroll
    for (int c = 0; c < 9; ++c) v[c] = c < NC ? mx[c < NC ? c : 0] : 0ull;
    v[9] = hi;
    v[10] = ~lo;   // the smallest as a largest
    v[11] = (unsigned long long)__double_as_longlong(err);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    links = __reduce_add_sync(0xffffffffu, links);
    thin = __reduce_add_sync(0xffffffffu, thin);
    if (lane == 0) {
        atomicAdd(&out->links[mu], (unsigned long long)links);
        atomicAdd(&out->thin[mu], (unsigned long long)thin);
    }
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        for (int o = 16; o > 0; o >>= 1) v[c] = umax64(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
        if (lane == 0) s_v[c][warp] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < 12) {
        unsigned long long t = 0ull;
        for (int w = 0; w < 8; ++w) t = umax64(t, s_v[threadIdx.x][w]);
        const int c = threadIdx.x;
        if (t != 0ull)
            atomicMax(c < 9 ? &out->comp[c] : c == 9 ? &out->hi[mu] : c == 10 ? &out->nlo[mu] : &out->err, t);
    }
}

// Component 6 of an R14 link alone: the pivot k is chosen in FP32 (where two
// of the |cc_k| agree to FP32 rounding either serves), the rest as in
// third_factor; 26 FP64 operations instead of 78.
__device__ __forceinline__ double2 r14_factor(const double2* m) {
    float2 u[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) u[c] = make_float2((float)m[c].x, (float)m[c].y);
    auto cross2 = [&](int a, int b, int c, int d) {
        const float x = u[a].x * u[b].x - u[a].y * u[b].y - (u[c].x * u[d].x - u[c].y * u[d].y);
        const float y = u[a].x * u[b].y + u[a].y * u[b].x - (u[c].x * u[d].y + u[c].y * u[d].x);
        return x * x + y * y;
    };
    const float n0 = cross2(1, 5, 2, 4), n1 = cross2(2, 3, 0, 5), n2 = cross2(0, 4, 1, 3);
    const int k = (n1 > n0) ? (n2 > n1 ? 2 : 1) : (n2 > n0 ? 2 : 0);
    const float best = fmaxf(n0, fmaxf(n1, n2));
    if (!(best > 1e-30f && best < 1e30f)) {   // FP32 range left
        double unused = 0.0;
        return third_factor<14>(m, 1, 1.0, unused);
    }
    const double2 a = k == 0 ? m[1] : k == 1 ? m[2] : m[0], b = k == 0 ? m[5] : k == 1 ? m[3] : m[4];
    const double2 c = k == 0 ? m[2] : k == 1 ? m[0] : m[1], d = k == 0 ? m[4] : k == 1 ? m[5] : m[3];
    const double2 mk = k == 0 ? m[6] : k == 1 ? m[7] : m[8];
    const double2 ck = zconj(zsub(zmul(a, b), zmul(c, d)));
    const double inv = 1.0 / (ck.x * ck.x + ck.y * ck.y);
    return make_double2((mk.x * ck.x + mk.y * ck.y) * inv, (mk.y * ck.x - mk.x * ck.y) * inv);
}

// fixed-point FP64 storage: v 2^(55 - e) rounded to an integer of at most 55
// bits, split into limbs of 28 bits (low limb balanced, see dslash_fx64.cuh),
// with integer instructions (|v| < 2^e, so the mantissa moves right)
__device__ __forceinline__ int2 fx_split(double v, int e) {
    const unsigned long long bits = abs_bits(v);
    const int field = (int)(bits >> 52);
    // left-aligned mantissa; bits to drop: 64 - 55 - (field - 1022) + e >= 9
    const unsigned long long m = (bits << 11) | 0x8000000000000000ull;
    const int sh = 9 + e + 1022 - field;
    long long q = 0;
    if (field > 0 && sh <= 63) q = (long long)((m >> sh) + ((m >> (sh - 1)) & 1ull));
    q = __double_as_longlong(v) < 0 ? -q : q;
    const int lo = (int)((unsigned)q << 4) >> 4;
    return make_int2((int)((q - lo) >> 28), lo);
}

// 16-bit fixed point: round to nearest of v / scale, clamped to +-32767 (NaN: -32767)
__device__ __forceinline__ short quantize(double v, double inv_scale) {
    const int q = abs_bits(v) > kInfBits ? -32767 : __double2int_rn(v * inv_scale);
    return (short)min(max(q, -32767), 32767);
}
__device__ __forceinline__ float4 store_pair(double2 a, double2 b, const double*, int, float2) {
    return make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
}
__device__ __forceinline__ short4 store_pair(double2 a, double2 b, const double* inv, int c, short2) {
    return make_short4(quantize(a.x, inv[c]), quantize(a.y, inv[c]), quantize(b.x, inv[c + 1]), quantize(b.y, inv[c + 1]));
}
__device__ __forceinline__ float2 store_one(double2 a, const double*, int, float2) {
    return make_float2((float)a.x, (float)a.y);
}
__device__ __forceinline__ short2 store_one(double2 a, const double* inv, int c, short2) {
    return make_short2(quantize(a.x, inv[c]), quantize(a.y, inv[c]));
}

// One pass over a field writes its FP64 copy, unless out_fx is null the
// fixed-point form of it, and unless the storage precision is FP64 (LC =
// double2) the storage copy. The FP64 pipe bounds it (the quantisation
// multiplies, z), so the fixed-point split uses integers only.
template <typename LC, int RECON>
__global__ void __launch_bounds__(256) pack_kernel(Geom g, const double2* __restrict__ canon, LinkScales sc,
                                                   double2* __restrict__ out64, int4* __restrict__ out_fx,
                                                   LC* __restrict__ out_lo) {
    constexpr int NC = RECON / 2;
    const unsigned V = 2u * (unsigned)g.vh;
    const int mu = blockIdx.y;
    const int fxe = sc.fx_exp[mu];
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
        const double2* src = canon + ((size_t)mu * V + i) * 9;
        const Site s = site_of(g, i);
        double2 m[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) m[c] = src[c];
        const size_t at = (size_t)(s.parity * 4 + mu) * 9 * g.vh + s.h;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            out64[at + (size_t)c * g.vh] = m[c];
            if (out_fx != nullptr) {
                const int2 re = fx_split(m[c].x, fxe), im = fx_split(m[c].y, fxe);
                out_fx[at + (size_t)c * g.vh] = make_int4(re.x, re.y, im.x, im.y);
            }
        }
        if constexpr (LinkPair<LC>::paired) {
            if (RECON == 14) m[6] = r14_factor(m);
            using P = typename LinkPair<LC>::V;
            LC* block = out_lo + (size_t)(s.parity * 4 + mu) * NC * g.vh;
#pragma unroll
            for (int p = 0; p < NC / 2; ++p)
                reinterpret_cast<P*>(block)[(size_t)p * g.vh + s.h] = store_pair(m[2 * p], m[2 * p + 1], sc.inv, 2 * p, LC{});
            if constexpr (NC & 1) block[(size_t)(NC - 1) * g.vh + s.h] = store_one(m[NC - 1], sc.inv, NC - 1, LC{});
        }
    }
}

__global__ void compress_kernel(Geom g, const double2* __restrict__ canon, int recon, int hop,
                                double inv_s, double* __restrict__ packed,
                                unsigned long long* err_bits) {
    const int nc = recon / 2;
    const long long V = 2ll * g.vh;
    double worst = 0.0;
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < 4 * V;
         w += (long long)gridDim.x * blockDim.x) {
        const int mu = (int)(w / V);
        const Site s = site_of(g, (unsigned)(w - mu * V));
        double2 m[9], enc[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) m[c] = canon[w * 9 + c];
        const int sg = (recon == 12) ? staggered_sign(g, s, mu, hop) : 1;
        worst = fmax(worst, encode(m, recon, sg, inv_s, enc));
        for (int c = 0; c < nc; ++c) {
            packed[w * recon + 2 * c] = enc[c].x;
            packed[w * recon + 2 * c + 1] = enc[c].y;
        }
    }
    if (err_bits != nullptr) atomic_max_nonneg(err_bits, worst);
}

__global__ void reconstruct_kernel(Geom g, const double* __restrict__ packed, int recon, int hop,
                                   double inv_s, double2* __restrict__ canon) {
    const int nc = recon / 2;
    const long long V = 2ll * g.vh;
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < 4 * V;
         w += (long long)gridDim.x * blockDim.x) {
        const int mu = (int)(w / V);
        const Site s = site_of(g, (unsigned)(w - mu * V));
        double2 m[9];
        for (int c = 0; c < nc; ++c)
            m[c] = make_double2(packed[w * recon + 2 * c], packed[w * recon + 2 * c + 1]);
        if (recon != 18) {
            double2 cc[3], f;
            cross_conj(m, cc);
            if (recon == 14) {
                f = m[6];
            } else {
                const int sg = staggered_sign(g, s, mu, hop);
                f = make_double2(sg > 0 ? inv_s : -inv_s, 0.0);
            }
            for (int c = 0; c < 3; ++c) m[6 + c] = zmul(f, cc[c]);
        }
        for (int c = 0; c < 9; ++c) canon[w * 9 + c] = m[c];
    }
}

unsigned grid_for(long long work, int per_sm = 32) {
    long long b = (work + 255) / 256;
    const long long cap = (long long)per_sm * device_sm_count();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

}  // namespace

cudaError_t launch_link_scan(const Geom& g, const double2* canon, int recon, int hop, double r12_inv_scale,
                             LinkScan* out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(*out), s);
    if (e != cudaSuccess) return e;
    const dim3 grid((grid_for(2ll * g.vh, 2) + 3) / 4, 4);
    switch (recon) {
        case 18: scan_kernel<18><<<grid, 256, 0, s>>>(g, canon, hop, r12_inv_scale, out); break;
        case 14: scan_kernel<14><<<grid, 256, 0, s>>>(g, canon, hop, r12_inv_scale, out); break;
        case 12: scan_kernel<12><<<grid, 256, 0, s>>>(g, canon, hop, r12_inv_scale, out); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_pack_links(const Geom& g, const double2* canon, int prec, int recon, const LinkScales& sc, void* out64,
                              void* out_fx, void* out_lo, cudaStream_t s) {
    const dim3 grid((grid_for(8ll * g.vh) + 3) / 4, 4);
    double2* o = (double2*)out64;
#define HISQ_PACK(LC, RECON) pack_kernel<LC, RECON><<<grid, 256, 0, s>>>(g, canon, sc, o, (int4*)out_fx, (LC*)out_lo)
    switch (prec * 100 + recon) {
        case HISQ_F64 * 100 + 18: HISQ_PACK(double2, 18); break;
        case HISQ_F32 * 100 + 18: HISQ_PACK(float2, 18); break;
        case HISQ_F32 * 100 + 14: HISQ_PACK(float2, 14); break;
        case HISQ_F32 * 100 + 12: HISQ_PACK(float2, 12); break;
        case HISQ_F16 * 100 + 18: HISQ_PACK(short2, 18); break;
        case HISQ_F16 * 100 + 14: HISQ_PACK(short2, 14); break;
        case HISQ_F16 * 100 + 12: HISQ_PACK(short2, 12); break;
        default: return cudaErrorInvalidValue;
    }
#undef HISQ_PACK
    return cudaGetLastError();
}

cudaError_t launch_compress_links(const Geom& g, const double2* canon, int recon, int hop,
                                  double r12_inv_scale, double* packed,
                                  unsigned long long* err_bits, cudaStream_t s) {
    compress_kernel<<<grid_for(8ll * g.vh), 256, 0, s>>>(g, canon, recon, hop, r12_inv_scale,
                                                         packed, err_bits);
    return cudaGetLastError();
}

cudaError_t launch_reconstruct_links(const Geom& g, const double* packed, int recon, int hop,
                                     double r12_inv_scale, double2* canon, cudaStream_t s) {
    reconstruct_kernel<<<grid_for(8ll * g.vh), 256, 0, s>>>(g, packed, recon, hop,
                                                            r12_inv_scale, canon);
    return cudaGetLastError();
}

}  // namespace hisq
