// Tables that depend on an architecture row and the axes only, built on the host and passed as kernel parameters
// (6.6 KB) that each CTA copies to shared memory, and the lookups the evaluation and search kernels make in them.
#pragma once

#include <stdint.h>

#include "eval_common.cuh"

namespace tune_dev {

constexpr int kMaxB = 32;  // blocks per SM supported by the tables
constexpr int kIparStride = 17;  // words per ipar row (16 grid positions and one of padding)

struct CtaTables {
    // (waves*slots)/(n_sm*G) by (B*-1, g position); +inf padding. Rows of 17 words, so that a
    // warp reading one g position of 32 rows (lane = row) touches 32 distinct banks.
    float ipar[kMaxB][kIparStride];
    float rcp[8];                    // 1 / IPC per class
    float rcpn[33];                  // 1 / n for n = 1..32 (axis-subset sizes; [0] unused)
    float hide[kMaxW + 1];           // max(1, W_sat / W*)
    float lane[32];                  // (32 * W_B) / T by t position
    int wb[32];                      // W_B = ceil(T / 32) by t position
    int gw[32];                      // G_W by t position (0 if T > max threads per block)
    unsigned char divt[kMaxW + 1][32];  // floor(w / W_B) by (w, t position)
    // g positions of ipar row b in increasing (value, g) order, backwards: the first is [15], so that the
    // highest set bit of a mask over these places is the next grid size; and the place of every g position,
    // four bits each
    unsigned char rperm[kMaxB][16];
    unsigned long long place[kMaxB];
    float iparmin[kMaxB];            // min of ipar row b over all axis grid sizes
    unsigned char rwarps[256];       // register-limited warps by R (Eq. 4, per-warp allocation; at most kMaxW)
    unsigned char rwbmax[256];       // largest W_B whose block fits the per-block register limit, by R, up to 255
    int cap_lo[4];                   // first capacity index allowed by carveout position c
    int order_safe;                  // 1: distinct ipar values of a row differ by more than 2^-21 relative
    int unit_shift;                  // log2 of the shared-memory allocation unit, or -1
};

// The tables from the launch parameters into shared memory (a word per thread and step).
__device__ __forceinline__ void copy_cta_tables(const CtaTables& src, CtaTables& ct)
{
    const uint32_t* s = reinterpret_cast<const uint32_t*>(&src);
    uint32_t* d = reinterpret_cast<uint32_t*>(&ct);
    for (int i = threadIdx.x; i < (int)(sizeof(CtaTables) / 4); i += blockDim.x) d[i] = s[i];
}

// q = floor(n / d) for 0 <= n < 2^25 and 1 <= d < 2^25: a single-precision estimate
// (within 2 of q) corrected with exact integer remainders.
__device__ __forceinline__ int udiv_small(int n, int d)
{
    int q = __float2int_rz(__fmul_rn((float)n, __frcp_rn((float)d)));
    int r = n - q * d;
    while (r < 0) {
        --q;
        r += d;
    }
    while (r >= d) {
        ++q;
        r -= d;
    }
    return q;
}

// G_S (Eq. 5) as smem_blocks(), starting the capacity search at the carveout's
// first admissible capacity (carveout position cp).
__device__ __forceinline__ int smem_blocks_from(const tune_arch& a, const CtaTables& ct, int s0, int cp)
{
    if (s0 > a.smem_block_max) return 0;
    const int need = s0 + a.smem_reserved_block;
    const int unit = a.smem_alloc_unit;
    const int s_alloc = ct.unit_shift >= 0 ? ((need + unit - 1) >> ct.unit_shift) << ct.unit_shift
                                           : ceil_div(need, unit) * unit;
    if (s_alloc == 0) return a.max_blocks_sm;
    for (int i = ct.cap_lo[cp]; i < a.n_smem_caps; ++i) {
        const int ci = a.smem_caps[i];
        if (ci >= s_alloc) return udiv_small(ci, s_alloc);
    }
    return 0;
}

// G_R (Eq. 4) for R registers and blocks of W_B warps (t position tp).
__device__ __forceinline__ int reg_blocks(const tune_arch& a, const CtaTables& ct, int R, int wb, int tp,
                                          int warps, int wbmax)
{
    if (R > a.regs_thread_max) return 0;
    if (R <= 0) return a.max_blocks_sm;
    if (a.reg_alloc_mode == 0) return wb > wbmax ? 0 : ct.divt[warps][tp];
    const long long rpb = (long long)ceil_div(R * 32 * wb, a.reg_alloc_unit) * a.reg_alloc_unit;
    return rpb > a.regs_block_max ? 0 : (int)(a.regs_sm / rpb);
}

}  // namespace tune_dev

namespace tune {

// The tables of a row and axes, from the calling thread's last few different ones where they are among them.
void eval_tables(const tune_arch& a, const tune_axes& x, tune_dev::CtaTables& out);

}  // namespace tune
