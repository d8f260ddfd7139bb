// Training forward of the surrogate on tcgen05: the inference kernel's roles (tc_mlp.cuh) in BF16, keeping
// what the backward pass reads: gelu'(z) of every layer (FP16, tiled, mlp::gprime_at) and the activations
// h = gelu(z) (BF16). act holds h itself, because it is also H1..H3 as the backward pass reads them: the
// MMA issuer copies each K chunk of act to global memory with a bulk tensor store while that chunk's MMAs
// read it, and waits for the copies to have read act before the epilogue may overwrite it.
//
// A training step has few units per SM (320 of 8,192 rows x 5 members on 152 SMs), so what counts is how
// long a unit takes by itself: sixteen warps serve each unit's epilogue, load their columns of the
// accumulator at once (which frees it for the next layer) and hand the layer's output over one K chunk at a
// time, so that the next layer's MMAs start while the later chunks are still being computed. 14 steps of
// 8,192 rows x 5 members: 2.17 -> 2.05 ms (2.21 with the inference kernel's split of the warps);
// 1.89 ms with the backward kernels' changes and the L2 policies (policy_evict_first), 1.72 ms with the
// small launches of a step merged into its large ones.
#pragma once

#include "tc_mlp.cuh"

namespace tcm {

// The head's backward pass over a slice of rows of one member (head_rows, head_sum): dy[i] =
// 2 (y[i] - lbl[i]) / n for the n labelled rows (0 past them), dZ4[i][j] = bf16(dy[i] * w5[j] *
// gelu'(Z4)[i][j]), and part[member][slice][j] = sum over the slice of dy[i] H4[i][j] (j < 256), of
// dy[i] (j = 256) and of (y[i] - lbl[i])^2 (j = 257).
constexpr int kHeadGroups = 8;          // row groups of 32 threads; group q takes rows q, q + 8, ...
constexpr int kHeadStride = kWid + 2;   // floats per slice of part
constexpr int kHeadRows = 64;           // rows of a slice (longer only where part would not hold them)

struct HeadArgs {
    const float* lbl;
    int n;
    __nv_bfloat16* dz;   // dZ4, [members][act_stride]
    float* part;
    int slices;          // per member
    int first;           // CTAs first .. gridDim.x - 1 do their own units' slices
};

struct TrainArgs {
    Args f;                     // the forward's arguments (rows < f.n are written to f.pred)
    __half* g_out[kLayers];     // gelu' of each layer, [members][act_stride]
    __nv_bfloat16* h4_out;      // H4, the same layout in rows of 256 (H1..H3 go through the map `th`)
    long long act_stride;
    HeadArgs head;
};

struct TrainControl {
    uint64_t w_full[Cfg<false>::stages], w_empty[Cfg<false>::stages];
    uint64_t x_full[2], act_free[2], acc_full[2], head_bar[2], drained[2], drain;
    uint64_t rdy[2][4];  // K chunk c of the chain's activations written by the epilogue
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(TrainControl) <= kControlBytes, "control block");

// What a bounded wait needs to give up: the launch's status word and the CTA's abort flag.
struct Abort {
    int* status;
    volatile int* flag;
};

// A persistent CTA's unit of ordinal jj (units < 2^28, so 32-bit division), tile by tile: the members of a
// tile share its input rows.
__device__ __forceinline__ Unit train_unit(int jj, int members)
{
    const unsigned u = blockIdx.x + (unsigned)jj * gridDim.x;
    const unsigned t = u / (unsigned)members;
    return {(int)t, (int)(u - t * (unsigned)members)};
}

// Training, t = gelu_tanh(z): gelu'(z) = (1 + t) / 2 + z / 2 (1 - t^2) K (1 + 3 C z^2); with
// 1 - t^2 = (1 - t)(1 + t) and a = (1 + t) / 2 it is a + (z K (1 + 3 C z^2)) (1 - t) a.
__device__ __forceinline__ uint32_t gelu_grad_half2(float2 z, float2 t)
{
    const float2 a = fma2(t, f2(0.5f), f2(0.5f));
    const float2 w = mul2(z, fma2(f2(3.0f * mlp::kGeluK * mlp::kGeluC), mul2(z, z), f2(mlp::kGeluK)));
    const float2 d = fma2(mul2(w, fma2(t, f2(-1.0f), f2(1.0f))), a, a);
    const __half2 d2 = __floats2half2_rn(d.x, d.y);
    return *reinterpret_cast<const uint32_t*>(&d2);
}

// Rows i0 + q, i0 + q + 8, ... < i1 of a slice, by the 32 threads of row group q (eight columns each, 16-byte
// accesses); the group's sums go to red[0 .. 257]. y, G4, H4, dZ: the member's. FRESH: y, G4 and H4 were
// written by this CTA (before a barrier). ROWS: rows whose loads are requested together.
template <bool FRESH, int ROWS>
__device__ __forceinline__ void head_rows(const float* y, const float* lbl, int n, const float* w5, const __half* G4,
                                          const __nv_bfloat16* H4, __nv_bfloat16* dZ, int i0, int i1, int q, int lane,
                                          float* red)
{
    const int j = 8 * lane;
    const float n_f = (float)n;
    float w[8];
    {
        const float4 a = *reinterpret_cast<const float4*>(w5 + j);
        const float4 b = *reinterpret_cast<const float4*>(w5 + j + 4);
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
    }
    float sh[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, sb = 0.0f, se = 0.0f;
#pragma unroll ROWS
    for (int i = i0 + q; i < i1; i += kHeadGroups) {
        float di = 0.0f;
        if (i < n) {
            const float e = (FRESH ? __ldcg(y + i) : y[i]) - lbl[i];
            di = 2.0f * e / n_f;
            se += e * e;
        }
        const long long o = (long long)i * kWid + j;
        const uint4* gp = reinterpret_cast<const uint4*>(G4 + mlp::gprime_at(i, j));
        const uint4* hp = reinterpret_cast<const uint4*>(H4 + o);
        const uint4 gv = FRESH ? __ldcg(gp) : __ldg(gp);
        const uint4 hv = FRESH ? __ldcg(hp) : __ldg(hp);
        const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, hw[4] = {hv.x, hv.y, hv.z, hv.w};
        uint32_t out[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float2 g = __half22float2(*reinterpret_cast<const __half2*>(&gw[t]));
            const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw[t]));
            const __nv_bfloat162 z = __floats2bfloat162_rn(di * w[2 * t] * g.x, di * w[2 * t + 1] * g.y);
            out[t] = *reinterpret_cast<const uint32_t*>(&z);
            sh[2 * t] = fmaf(di, h.x, sh[2 * t]);
            sh[2 * t + 1] = fmaf(di, h.y, sh[2 * t + 1]);
        }
        *reinterpret_cast<uint4*>(dZ + o) = make_uint4(out[0], out[1], out[2], out[3]);
        sb += di;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) red[j + c] = sh[c];
    if (j == 0) {
        red[kWid] = sb;
        red[kWid + 1] = se;
    }
}

// The row groups' sums (red[group][258], after a barrier), added in group order, by 256 threads.
__device__ __forceinline__ void head_sum(const float* red, int tid, float* part)
{
    for (int c = tid; c < kHeadStride; c += 32 * kHeadGroups) {
        float v = red[c];
#pragma unroll
        for (int g = 1; g < kHeadGroups; ++g) v += red[g * kHeadStride + c];
        part[c] = v;
    }
}

// Registers that an asynchronous TMEM load filled, after its wait: no use of them moves above it.
template <int N>
__device__ __forceinline__ void pin(uint32_t (&r)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}

// Starts the load of 16 consecutive accumulator columns of this thread's TMEM lane (row).
__device__ __forceinline__ void tmem_ld16_start(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// A warp's share of K chunk c of a layer's output is written: make it visible to the tensor cores
// and tell the MMA issuer.
__device__ __forceinline__ void chunk_done(uint64_t* bar, int lane)
{
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

// A warp's 64 of a layer's 256 accumulator columns, thread = row: per 16 columns 32 bytes of gelu' and BF16
// h. The head's columns are consecutive (the sum over them is returned); a hidden layer's are a quarter of
// each K chunk (rdy[c]: chunk c written). g_row: gelu' of the row at column 0 (16-column blocks 2,048
// elements apart); h_row: H4 of the row.
template <bool HEAD>
__device__ __forceinline__ float train_rows(uint32_t tlane, const float* bias, const float* w5, uint8_t* act, int r, int cq,
                                            int lane, __half* g_row, __nv_bfloat16* h_row, uint64_t* bar, uint64_t* rdy,
                                            uint32_t acc_ph, const Abort& ab, bool& ok)
{
    // the warp's 16-column block b: of the head, consecutive; else one of every K chunk
    auto col = [&](int b) { return HEAD ? 64 * cq + 16 * b : 64 * b + 16 * cq; };
    float bb[16], ww[16];
    ld16(bias + col(0), bb);
    if (HEAD) ld16(w5 + col(0), ww);
    ok = wait_bar_warp(bar, acc_ph, ab.status, ab.flag);
    if (!ok) return 0.0f;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t v[4][16];
#pragma unroll
    for (int b = 0; b < 4; ++b) tmem_ld16_start(tlane + col(b), v[b]);
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int b = 0; b < 4; ++b) pin(v[b]);
    float y = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        uint32_t w[8], gd[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 z = fma2(as_pair(v[b][2 * i], v[b][2 * i + 1]), f2(1.0f), make_float2(bb[2 * i], bb[2 * i + 1]));
            const float2 t = gelu_tanh(z);
            float2 h = fma2(z, t, z);
            h = mul2(h, f2(0.5f));  // h itself (2 h halved, exact): act, H and the head all take h
            gd[i] = gelu_grad_half2(z, t);
            w[i] = pack_bf16(h.x, h.y);
            if (HEAD) {
                y = fmaf(ww[2 * i], h.x, y);
                y = fmaf(ww[2 * i + 1], h.y, y);
            }
        }
        if (b < 3) {
            ld16(bias + col(b + 1), bb);
            if (HEAD) ld16(w5 + col(b + 1), ww);
        }
        st_global_v8<!HEAD>(g_row + col(b) * 128, gd);  // (gelu'(Z4) is read next)
        if (HEAD) {
            st_global_v8(h_row + col(b), w);
        } else {  // 16 columns = two 16-byte units
            uint8_t* base = act + b * kChunkA;
            st_shared_v4(base + swz(r, 2 * cq), w[0], w[1], w[2], w[3]);
            st_shared_v4(base + swz(r, 2 * cq + 1), w[4], w[5], w[6], w[7]);
            chunk_done(rdy + b, lane);
        }
    }
    return y;
}

// grid: min(SMs, units) persistent CTAs; CTA b runs units b, b + gridDim.x, ...; its j-th unit goes to chain
// j % 2. Unit u = (tile u / members, member u % members). 96 registers per thread, as mlp_infer_kernel's
// launch (18 warps: five on the fullest sub-partition).
__global__ void __maxnreg__(96) mlp_train_kernel(const __grid_constant__ CUtensorMap tx,
                                                 const __grid_constant__ CUtensorMap tw1,
                                                 const __grid_constant__ CUtensorMap tw,
                                                 const __grid_constant__ CUtensorMap th,
                                                 const __grid_constant__ TrainArgs t)
{
    using C = Cfg<false>;
    const Args& g = t.f;
    extern __shared__ uint8_t smem_raw[];

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ring = smem + 2 * C::act_bytes;
    TrainControl& ctl = *reinterpret_cast<TrainControl*>(ring + C::stages * kChunkW);
    // the warp number through a shuffle, so that the roles' branches and the MMA issuer's descriptor
    // arithmetic compile as warp-uniform
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int units = (int)g.units;
    const int my_units = units > (int)blockIdx.x ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    volatile int* abort_v = &ctl.abort_flag;

    pdl::grid_dep_enter();  // launched after the batch gather in a training step
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tc::sa(&ctl.tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (threadIdx.x == 32) {
        for (int i = 0; i < C::stages; ++i) {
            tc::mbar_init(&ctl.w_full[i], 1);
            tc::mbar_init(&ctl.w_empty[i], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&ctl.x_full[s], 1);
            tc::mbar_init(&ctl.act_free[s], 1);
            tc::mbar_init(&ctl.acc_full[s], 1);
            tc::mbar_init(&ctl.drained[s], kEpiWarps);
            tc::mbar_init(&ctl.head_bar[s], 3 * kEpiWarps / 4);
            for (int c = 0; c < 4; ++c) tc::mbar_init(&ctl.rdy[s][c], kEpiWarps);
        }
        tc::mbar_init(&ctl.drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        ctl.abort_flag = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = ctl.tmem_base;

    if (warp == 0) {
        // ---- producer: per unit pair, layer by layer, chain by chain (the MMA order) ----
        if (lane == 0) {
            int st = 0, issued = 0;      // ring stage of the next weight chunk; stages filled at least once
            uint32_t wph = 1;            // parity of w_empty for it (the first pass over the ring does not wait)
            int x_last[2] = {-1, -1};    // last unit whose input rows were requested, per chain
            bool ok = true;
            for (int j = 0; j < my_units && ok; j += 2) {
                const Unit un[2] = {train_unit(j, g.members), train_unit(j + 1, g.members)};
                const int ns = min(2, my_units - j);
                for (int l = 0; l < kLayers && ok; ++l) {
#pragma unroll 1
                    for (int s = 0; s < ns && ok; ++s) {
                        const int tile = s ? un[1].tile : un[0].tile, mem = s ? un[1].mem : un[0].mem;
                        if (l == 0) {
                            // the chain's buffer is free once the unit two before finished its MMAs
                            if (j >= 2 && !(ok = wait_bar(&ctl.act_free[s], (uint32_t)(((j - 2) >> 1) & 1), g.status,
                                                          abort_v)))
                                break;
                            uint8_t* act = smem + s * C::act_bytes;
                            tc::mbar_expect_tx(&ctl.x_full[s], C::chunks(0) * kChunkA);
                            for (int c = 0; c < C::chunks(0); ++c)
                                tma_load_2d(act + c * kChunkA, &tx, c * 16, tile * kRows, &ctl.x_full[s]);
                            x_last[s] = j + s;
                        }
                        for (int c = 0; c < C::chunks(l); ++c) {
                            if (!(ok = wait_bar(&ctl.w_empty[st], wph, g.status, abort_v))) break;
                            tc::mbar_expect_tx(&ctl.w_full[st], kChunkW);
                            // maps address 8-byte elements: 16 per 128-byte K chunk
                            if (l == 0)
                                tc::tma_load_3d(ring + st * kChunkW, &tw1, c * 16, 0, mem, &ctl.w_full[st]);
                            else
                                tma_load_4d(ring + st * kChunkW, &tw, c * 16, 0, l - 1, mem, &ctl.w_full[st]);
                            issued = max(issued, st + 1);
                            if (++st == C::stages) {
                                st = 0;
                                wph ^= 1;
                            }
                        }
                    }
                }
            }
            if (!ok) {
                // let the copies that may still be in flight land before the CTA exits: the last fill
                // of every stage used (those before `st` belong to the current pass over the ring)
                for (int q = 0; q < issued; ++q)
                    tc::mbar_wait(&ctl.w_full[q], q < st ? wph ^ 1 : wph, g.status);
                for (int s = 0; s < 2; ++s)
                    if (x_last[s] >= 0) tc::mbar_wait(&ctl.x_full[s], (uint32_t)((x_last[s] >> 1) & 1), g.status);
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer: the whole warp walks the loop (uniform descriptors and waits), one
        // elected lane issues ----
        const bool leader = elect_one();
        int st = 0;
        uint32_t wph = 0;
        bool ok = true;
        const uint64_t b_ring = tc::sdesc(ring);
        const uint64_t h_policy = policy_evict_first();  // H1..H3 are read last of all, by the weight gradients
        for (int j = 0; j < my_units && ok; j += 2) {
            const Unit un[2] = {train_unit(j, g.members), train_unit(j + 1, g.members)};
            const int ns = min(2, my_units - j);
            for (int l = 0; l < kLayers && ok; ++l) {
#pragma unroll 1
                for (int s = 0; s < ns && ok; ++s) {
                    if (l == 0) {
                        // the unit's input rows, and the chain's accumulator read by the last unit's head
                        if (!(ok = wait_bar_warp(&ctl.x_full[s], (uint32_t)((j >> 1) & 1), g.status, abort_v))) break;
                        if (j > 0 &&
                            !(ok = wait_bar_warp(&ctl.drained[s], (uint32_t)(((j >> 1) - 1) & 1), g.status, abort_v)))
                            break;
                    }
                    const uint8_t* act = smem + s * C::act_bytes;
                    const uint32_t d = tmem + (uint32_t)(s * kWid);
                    uint64_t a = tc::sdesc(act);  // addresses in the descriptors count 16-byte units
                    for (int c = 0; c < C::chunks(l); ++c, a += kChunkA >> 4) {
                        if (!(ok = wait_bar_warp(&ctl.w_full[st], wph, g.status, abort_v))) break;
                        // chunk c of the previous layer's output (ordinal 3 (j / 2) + l - 1 of its barrier)
                        if (l > 0 && !(ok = wait_bar_warp(&ctl.rdy[s][c], (uint32_t)(((j >> 1) + l - 1) & 1), g.status,
                                                          abort_v)))
                            break;
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        const uint64_t b = b_ring + (uint64_t)(st * (kChunkW >> 4));
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                tc::mma_bf16(d, a + kk * 2, b + kk * 2, tc::idesc_bf16(kRows, kWid), (c | kk) != 0);
                            tc::mma_commit(&ctl.w_empty[st]);
                            // H of layer l - 1 (BF16 h, rows of this unit's tile) is copied to global memory
                            // by the tensor-store unit while the MMAs read it
                            if (l > 0)
                                tma_store_4d(&th, act + c * kChunkA, c * 16, (s ? un[1].tile : un[0].tile) * kRows,
                                             s ? un[1].mem : un[0].mem, l - 1, h_policy);
                        }
                        __syncwarp();
                        if (++st == C::stages) {
                            st = 0;
                            wph ^= 1;
                        }
                    }
                    if (!ok) break;
                    if (leader) {
                        if (l > 0) {  // the epilogue rewrites act after acc_full
                            bulk_commit();
                            bulk_wait_read();
                        }
                        tc::mma_commit(&ctl.acc_full[s]);
                        if (l == kLayers - 1) tc::mma_commit(&ctl.act_free[s]);
                    }
                    __syncwarp();
                }
            }
        }
        if (leader) {
            bulk_wait_all();
            tc::mma_commit(&ctl.drain);  // arrives when every MMA issued above has completed
            tc::mbar_wait(&ctl.drain, 0, g.status);
        }
        __syncwarp();
    } else {
        // ---- epilogue: all sixteen warps serve the chains in the MMA issue order; warp = (TMEM lane
        // quarter q, quarter cq of every K chunk's columns; of the head's: 64 columns) ----
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const int r = q * 32 + lane;  // row in the tile where thread = accumulator row
        const Abort ab{g.status, abort_v};
        bool ok = true;
        for (int j = 0; j < my_units && ok; j += 2) {
            const Unit u0 = train_unit(j, g.members), u1 = train_unit(j + 1, g.members);
            const int ns = min(2, my_units - j);
            for (int l = 0; l < kLayers && ok; ++l) {
#pragma unroll 1
                for (int s = 0; s < ns && ok; ++s) {
                    const int tile = s ? u1.tile : u0.tile, mem = s ? u1.mem : u0.mem, row = tile * kRows + r;
                    const float* prm = g.master + mem * g.P;
                    const float* bias = prm + g.off_b[l];
                    uint8_t* act = smem + s * C::act_bytes;
                    const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(s * kWid);
                    const uint32_t acc_ph = (uint32_t)(l & 1);  // of ordinal 4 (j / 2) + l
                    __half* g_row = t.g_out[l] + (long long)mem * t.act_stride + mlp::gprime_at(row, 0);
                    if (l == kLayers - 1) {
                        // (H4 has no act copy: stored from here; H1..H3 leave from act, see the MMA issuer)
                        __nv_bfloat16* h_row = t.h4_out + (long long)mem * t.act_stride + (long long)row * kWid;
                        const float yh = train_rows<true>(tlane, bias, prm + g.off_w5, act, r, cq, lane, g_row, h_row,
                                                          &ctl.acc_full[s], nullptr, acc_ph, ab, ok);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                        // the other column quarters' sums for quarter 0, in the chain's second K chunk: its
                        // MMAs are done, and the next unit writes it only after quarter 0 has arrived on
                        // `drained` below
                        float* part = reinterpret_cast<float*>(act + kChunkA);
                        if (cq > 0) {
                            part[(cq - 1) * kRows + r] = yh;
                            __syncwarp();
                            if (lane == 0) {
                                mbar_arrive(&ctl.head_bar[s]);
                                mbar_arrive(&ctl.drained[s]);
                            }
                        } else {
                            if (!(ok = wait_bar_warp(&ctl.head_bar[s], (uint32_t)((j >> 1) & 1), g.status, abort_v))) break;
                            const float sum = ((yh + part[r]) + part[kRows + r]) + part[2 * kRows + r];
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&ctl.drained[s]);
                            if (row < g.n)
                                g.pred[(long long)mem * g.pred_stride + row] = sum + prm[g.off_b5];
                        }
                    } else {
                        train_rows<false>(tlane, bias, nullptr, act, r, cq, lane, g_row, nullptr, &ctl.acc_full[s],
                                          ctl.rdy[s], acc_ph, ab, ok);
                    }
                }
            }
        }
        // The head's backward pass of this CTA's units, while the CTAs with one unit more run theirs: two
        // slices (128 rows) at a time, warps 2-9 and 10-17 one each, sums through the activation buffers
        // (after an abort the results are as useless as the forward's, but every access is in bounds and
        // every warp is at the barriers).
        const HeadArgs& hd = t.head;
        if ((int)blockIdx.x >= hd.first) {
            const int grp = (warp - 2) >> 3, hq = (warp - 2) & 7;
            float* red = reinterpret_cast<float*>(smem) + grp * kHeadGroups * kHeadStride;
            named_barrier(1, 32 * kEpiWarps);
            for (int j = 0; j < my_units; ++j) {
                const Unit u = train_unit(j, g.members);
                const int i0 = u.tile * kRows + grp * kHeadRows;
                const long long base = (long long)u.mem * t.act_stride;
                head_rows<true, 2>(g.pred + (long long)u.mem * g.pred_stride, hd.lbl, hd.n, g.master + u.mem * g.P + g.off_w5,
                                t.g_out[kLayers - 1] + base, t.h4_out + base, hd.dz + base, i0, i0 + kHeadRows, hq, lane,
                                red + hq * kHeadStride);
                named_barrier(2 + grp, 32 * kHeadGroups);
                head_sum(red, 32 * hq + lane, hd.part + ((long long)u.mem * hd.slices + i0 / kHeadRows) * kHeadStride);
                named_barrier(2 + grp, 32 * kHeadGroups);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
}

}  // namespace tcm
