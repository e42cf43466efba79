// Block partials and their sums, in a fixed order (deterministic).
//
// Every block writes one partial per reduced value to partials[value * slots +
// blockIdx.x]. In the vector kernels, and the Dslash of few blocks (slots =
// kMaxRedBlocks), it then fences and bumps a counter; the block that arrives
// last sums the partials of every value in a fixed order (one warp per value,
// lane-strided, then a fixed shuffle tree), resets the counter for the next
// launch and runs the finish logic. A Dslash of many blocks (slots =
// kDeferSlots) leaves both to red_finish_kernel.
#pragma once

#include "hisq_internal.cuh"

namespace hisq {

template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename R>
__device__ __forceinline__ R warp_max(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// N per-lane values (N a power of two <= 32) reduced over the warp together:
// every exchange halves the values a lane carries, so 8 values take 9 shuffles
// instead of 40. The result is value multi_index<N>(lane), in all lanes that
// agree in the top log2(N) bits of the lane number; fixed order.
template <int N>
__device__ __forceinline__ int multi_index(int lane) {
    return N == 1 ? 0 : lane / (32 / N);
}
template <int N, typename R, typename Op>
__device__ __forceinline__ R warp_multi(R (&v)[N], Op op) {
    const int lane = threadIdx.x & 31;
    int mask = 16;
#pragma unroll
    for (int w = N / 2; w >= 1; w >>= 1, mask >>= 1) {
        const bool up = lane & mask;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const R send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, mask));
        }
    }
    R t = v[0];
#pragma unroll
    for (; mask >= 1; mask >>= 1) t = op(t, __shfl_xor_sync(0xffffffffu, t, mask));
    return t;
}

// Signals arrival of this block; true in the block that arrived last.
__device__ __forceinline__ bool last_block_arrive(unsigned int* counter, unsigned int nblocks) {
    __shared__ unsigned int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const unsigned int prev = atomicAdd(counter, 1u);
        s_last = (prev == nblocks - 1u) ? 1u : 0u;
    }
    __syncthreads();
    return s_last != 0u;
}

// In the last block: out[v] = sum (or max, when is_max(v)) over slots of
// partials[v][0 .. nslots). Must be called by all threads of the block.
template <int U = 1, typename IsMax>
__device__ __forceinline__ void finish_values(const RedScratch& red, int nvals, int nslots,
                                              IsMax is_max, double* out_smem) {
    __threadfence();
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nthreads = blockDim.x * blockDim.y;
    const int warp = tid >> 5, lane = tid & 31, nwarps = nthreads >> 5;
    for (int v = warp; v < nvals; v += nwarps) {
        const double* src = red.partials + (size_t)v * kMaxRedBlocks;
        const bool mx = is_max(v);
        double acc = 0.0;
        if (U > 1 && nslots > 64) {
            // U loads in flight per lane: up to 4096 slots are summed while the
            // rest of the GPU waits
            for (int i0 = lane; i0 < nslots; i0 += 32 * U) {
                double t[U];
#pragma unroll
                for (int u = 0; u < U; ++u) t[u] = i0 + 32 * u < nslots ? __ldcg(src + i0 + 32 * u) : 0.0;
#pragma unroll
                for (int u = 0; u < U; ++u) acc = mx ? fmax(acc, t[u]) : acc + t[u];
            }
        } else {
            for (int i = lane; i < nslots; i += 32) {
                const double t = __ldcg(src + i);
                acc = mx ? fmax(acc, t) : acc + t;
            }
        }
        acc = mx ? warp_max(acc) : warp_sum(acc);
        if (lane == 0) out_smem[v] = acc;
    }
    if (tid == 0) *red.counter = 0u;
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Finish logic shared by the Dslash and vector kernels
// ---------------------------------------------------------------------------

// An rhs moves (takes part in alpha/beta updates) while active and not frozen.
__device__ __forceinline__ bool moving(const CgScalars* cg, int k) {
    return cg->active[k] && !cg->frozen[k];
}

// The scalars of rhs k that the finishes read, loaded together (one latency
// instead of one for each that follows a branch).
struct FinState {
    int moves, stall;
    double rr, rr_rel, freeze2, alpha_max;
};
__device__ __forceinline__ FinState fin_load(const CgScalars* cg, int k) {
    FinState f = {};
    if (cg == nullptr) return f;
    const int act = cg->active[k], frz = cg->frozen[k];
    f.stall = cg->stall[k];
    f.rr = cg->rr[k];
    f.rr_rel = cg->rr_rel[k];
    f.freeze2 = cg->freeze2;
    f.alpha_max = cg->alpha_max;
    f.moves = act && !frz;
    return f;
}

// pAp -> alpha_k = rr_k / pAp_k for a moving rhs k. A non-finite pAp is an
// error; pAp <= 0 means the low-precision iteration lost A-conjugacy: alpha = 0
// and this iteration restarts the rhs from p = r (beta = 0).
__device__ __forceinline__ void finish_cg_alpha(CgScalars* cg, int k, double pAp, const FinState& f) {
    double alpha = 0.0;
    if (f.moves) {
        if (!isfinite(pAp)) {
            atomicOr(&cg->flags, kFlagNaN);
        } else if (!(pAp > 0.0) || !(f.rr <= f.alpha_max * pAp)) {
            // pAp <= 0, or alpha above 1/lambda_min: the low-precision
            // iteration lost conjugacy; restart this rhs from p = r
            cg->stall[k] = 1;
        } else {
            alpha = f.rr / pAp;
        }
    }
    cg->pAp[k] = pAp;
    cg->alpha[k] = alpha;
}

// rr' -> beta_k = rr'_k / rr_k, rr_k = rr'_k for a moving rhs; freezes an rhs
// whose residual fell by more than freeze2 since the last reliable update.
__device__ __forceinline__ void finish_cg_beta(CgScalars* cg, int k, double rr_new, const FinState& f) {
    double beta = 0.0;
    if (f.moves) {
        if (!isfinite(rr_new)) {
            atomicOr(&cg->flags, kFlagNaN);
        } else {
            if (f.stall) {
                cg->stall[k] = 0;
                cg->restarts[k] += 1;
            } else if (f.rr > 0.0) {
                beta = rr_new / f.rr;
            }
            cg->rr[k] = rr_new;
            if (rr_new <= f.freeze2 * f.rr_rel) cg->frozen[k] = 1;
        }
    }
    cg->beta[k] = beta;
}

// FP64 true residual of rhs k (|r|^2 and max |r_i|): record it, retire the rhs
// if it meets tol2 * |b|^2, pick the next scale.
__device__ __forceinline__ void finish_reliable(CgScalars* cg, int k, double nrm, double mx, double tol2) {
    // The search direction p is kept across the update while the
    // iterated residual still describes the true one. Once the true
    // residual is 10x (in norm) above the iterated one, the iteration has
    // run into its rounding floor and p no longer belongs to this
    // residual; a frozen rhs skipped its last p update. Both restart
    // from p = r.
    const double sc = cg->scale[k];
    const double iterated = cg->rr[k] / (sc * sc);
    cg->reset_p[k] = (nrm > 100.0 * iterated || cg->frozen[k]) ? 1 : 0;
    cg->rr_true[k] = nrm;
    cg->rmax[k] = mx;
    const int better = isfinite(nrm) && (!cg->have_best[k] || nrm < cg->rr_best[k]);
    cg->keep[k] = better;
    if (better) {
        cg->rr_best[k] = nrm;
        cg->have_best[k] = 1;
    }
    if (!isfinite(nrm)) {
        atomicOr(&cg->flags, kFlagNaN);
        cg->active[k] = 0;
    } else if (cg->active[k] && nrm <= tol2 * cg->bb[k]) {
        cg->active[k] = 0;
    }
    cg->scale_old[k] = cg->scale[k];
    cg->scale[k] = (mx > 0.0 && isfinite(mx)) ? 1.0 / mx : 1.0;
}

// The reduced value(s) of rhs k as the finish of a reduction with nv values
// per rhs: v0, and v1 (the maximum) with nv = 2.
__device__ __forceinline__ void finish_rhs(int finish, CgScalars* cg, double* out, int k, int nv, double v0, double v1,
                                           double tol2, const FinState& f) {
    if (finish == FIN_CG_ALPHA) {
        finish_cg_alpha(cg, k, v0, f);
    } else if (finish == FIN_CG_BETA) {
        finish_cg_beta(cg, k, v0, f);
    } else if (finish == FIN_RELIABLE) {
        finish_reliable(cg, k, v0, v1, tol2);
    } else if (out != nullptr) {
        out[k * nv] = v0;
        if (nv == 2) out[k * nv + 1] = v1;
    }
}

}  // namespace hisq
