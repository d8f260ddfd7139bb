// Host side of eval_tables.cuh.
#include "eval_tables.cuh"

#include <string.h>

#include <algorithm>
#include <limits>

using namespace tune_dev;

namespace {

constexpr int kKept = 8;  // results kept per thread (the rows of one tune_eval_archs call)

// The tables of an architecture row and axes (IEEE single-precision divisions and multiplications, each
// rounded to nearest as __fdiv_rn / __fmul_rn round them on the device).
void host_cta_tables(const tune_arch& a, const tune_axes& x, CtaTables& ct)
{
    memset(&ct, 0, sizeof(ct));
    const float inf = std::numeric_limits<float>::infinity();
    for (int b = 0; b < kMaxB; ++b)
        for (int g = 0; g < 16; ++g) {
            float v = inf;
            if (b < a.max_blocks_sm && g < x.n_g) {
                const int slots = a.n_sm * (b + 1), G = x.g[g];
                const int waves = (G + slots - 1) / slots;
                v = (float)(waves * slots) / (float)(a.n_sm * G);
            }
            ct.ipar[b][g] = v;
        }
    for (int w = 0; w <= kMaxW; ++w)
        for (int t = 0; t < 32; ++t) {
            const int wb = t < x.n_t ? (x.t[t] + 31) / 32 : 1;
            ct.divt[w][t] = (unsigned char)(w / wb);
        }
    // With distinct ipar values more than 2^-21 apart, X * v keeps their order strictly for every X > 0 (no
    // underflow), so a walk in perm order meets equal costs only from equal values, in increasing g (and index)
    // order.
    ct.order_safe = 1;
    const int u = a.smem_alloc_unit;
    ct.unit_shift = (u & (u - 1)) == 0 ? __builtin_ctz((unsigned)u) : -1;
    for (int b = 0; b < kMaxB; ++b) {
        float mn = inf;
        for (int g = 0; g < x.n_g; ++g) mn = std::min(mn, ct.ipar[b][g]);
        ct.iparmin[b] = mn;
        unsigned char ord[16] = {};
        for (int g = 0; g < x.n_g; ++g) {
            const float v = ct.ipar[b][g];
            int j = g;
            while (j > 0 && ct.ipar[b][ord[j - 1]] > v) {
                ord[j] = ord[j - 1];
                --j;
            }
            ord[j] = (unsigned char)g;
        }
        for (int r = 0; r < x.n_g; ++r) {
            ct.rperm[b][15 - r] = ord[r];
            ct.place[b] |= (unsigned long long)(15 - r) << (4 * ord[r]);
        }
        for (int r = 0; r + 1 < x.n_g; ++r) {
            const float v1 = ct.ipar[b][ord[r]], v2 = ct.ipar[b][ord[r + 1]];
            const volatile float gap = v2 - v1, tol = v1 * 0x1p-21f;  // two roundings, no fused form
            if (v2 != v1 && gap <= tol) ct.order_safe = 0;
        }
    }
    for (int t = 0; t < 32; ++t) {
        int wb = 1, gw = 0;
        float ln = 1.0f;
        if (t < x.n_t) {
            const int T = x.t[t];
            wb = (T + 31) / 32;
            gw = T <= a.max_threads_block ? std::min(a.max_blocks_sm, a.max_warps_sm / wb) : 0;
            ln = (float)(32 * wb) / (float)T;
        }
        ct.wb[t] = wb;
        ct.gw[t] = gw;
        ct.lane[t] = ln;
    }
    for (int w = 0; w <= kMaxW; ++w) ct.hide[w] = std::max(1.0f, w > 0 ? (float)a.w_sat / (float)w : 1.0f);
    for (int c = 0; c < 8; ++c) ct.rcp[c] = c < TUNE_NCLASS ? 1.0f / a.ipc[c] : 0.0f;
    for (int n = 1; n <= 32; ++n) ct.rcpn[n] = 1.0f / (float)n;
    for (int c = 0; c < 4; ++c) {
        const long long need = c < x.n_c ? (long long)x.c[c] * a.smem_caps[a.n_smem_caps - 1] : 0;
        int i = 0;
        while (i < a.n_smem_caps && 100LL * a.smem_caps[i] < need) ++i;
        ct.cap_lo[c] = i;
    }
    for (int R = 0; R < 256; ++R) {
        int warps, wbmax;
        reg_params(a, R, warps, wbmax);
        ct.rwarps[R] = (unsigned char)warps;
        // (a block of more than kMaxW warps has G_W = 0, so the limit beyond 255 does not matter)
        ct.rwbmax[R] = (unsigned char)std::min(wbmax, 255);
    }
}

}  // namespace

// From the calling thread's last kKept different rows and axes where they are
// among them (compared byte for byte).
void tune::eval_tables(const tune_arch& a, const tune_axes& x, CtaTables& out)
{
    struct Entry {
        tune_arch a;
        tune_axes x;
        CtaTables t;
    };
    static thread_local Entry kept[kKept];
    static thread_local int n_kept = 0, oldest = 0;
    for (int i = 0; i < n_kept; ++i)
        if (memcmp(&kept[i].a, &a, sizeof(tune_arch)) == 0 && memcmp(&kept[i].x, &x, sizeof(tune_axes)) == 0) {
            out = kept[i].t;
            return;
        }
    Entry& e = kept[n_kept < kKept ? n_kept++ : (oldest++ % kKept)];
    e.a = a;
    e.x = x;
    host_cta_tables(e.a, e.x, e.t);
    out = e.t;
}
