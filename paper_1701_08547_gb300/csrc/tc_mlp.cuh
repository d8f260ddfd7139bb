// Fused surrogate inference on tcgen05: one persistent CTA per SM pushes
// 128-row tiles of feature rows through whole ensemble members (four hidden
// layers and the head) without writing activations to global memory. (The
// training forward, tc_mlp_train.cuh, shares the helpers of this file.)
//
// Work unit = (member, tile of 128 rows). A CTA runs two units at a time, one
// per "chain": each chain owns an activation buffer in shared memory and a
// 256-column FP32 accumulator in tensor memory. Layer l of a unit is
//   MMA:      acc = act . W_l^T              (tcgen05.mma, operands in smem)
//   epilogue: act = q(2 gelu(acc * s + b))   (tcgen05.ld, CUDA cores, smem stores)
// and the MMA issuer alternates the chains layer by layer, so one chain's
// epilogue runs while the other chain's MMAs occupy the tensor cores.
//
// Roles (640 threads): warp 0 streams weights (and each unit's input rows)
// with TMA through a ring of 32 KB stages (all 256 output rows of a 128-byte
// K chunk; the tensor maps address 8-byte elements, the bytes and their
// 128-byte swizzle being the same for BF16 and E4M3 data); warp 1 issues the MMAs; warps 4-11
// and 12-19 run the epilogues of the two chains (four warps per half of the columns, one per
// TMEM lane quarter).
//
// What bounds it (2^20 rows x 5 members): an epilogue's 32,768 tanh take the multi-function units 2,048
// cycles, a layer's MMAs take the tensor cores 2,048; a chain alternates the two, in about 6,000 cycles per
// layer of both chains. What the rest goes to is not separated: the waits between the two (100 cycles each
// alone, 200-350 among busy epilogue warps), or the path to shared memory and L1, which carries the MMAs'
// operand reads in 35 % of the cycles, the epilogues' accesses in 43 % (30 of them parameter loads that hit L1)
// and the TMA's writes in 24 % (counters, 131,072 rows). BF16 2.25 -> 1.84 ms, E4M3 (100,003 rows) 0.192 ->
// 0.174 ms, against a kernel with the
// same roles whose every thread divided 64-bit unit numbers and arrived on the barriers by itself, whose
// sixteen epilogue warps served the chains in turn with thread = row, and whose single issuing lane
// could not keep its descriptors in uniform registers (700-900 cycles per chunk of four MMAs, now
// 480-600). Not kept (best of ten passes, this kernel 1.79 ms): sixteen warps per epilogue with the accumulator
// loaded at once and handed over
// chunk by chunk (1.96 ms here, but the better form for training's few units, tc_mlp_train.cuh); two
// N = 128 halves (2.26 ms: the A operand is read twice from shared memory); twelve warps of 72
// registers per chain (1.90 ms); no register split (1.85 ms, spills).
//
// The epilogue stores 2 gelu(z) = z (1 + tanh u), one operation fewer than
// gelu itself, and the next layer (or the head) takes half its accumulator.
// In BF16 this is exact: doubling commutes with rounding, so the results are
// those of storing gelu(z).
//
// Precision: layer 1 (K = 64) is BF16 x BF16 in both variants; GELU is
// evaluated in FP32. The BF16 variant keeps layers 2-4 in BF16; the FP8
// variant stores E4M3 codes of 2 h (activation scale 1/2) and W2..W4 as E4M3
// codes with one scale per matrix, and runs layers 2-4 with kind::f8f6f4.
// The head takes the FP32 values 2 h4 and sums in FP32.
//
// Every wait is bounded; on timeout the kernel sets status bit 2, stops
// issuing work, waits (bounded) for the copies and MMAs it issued, frees its
// tensor memory and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include "f32x2.cuh"
#include "gelu.cuh"
#include "pdl.cuh"
#include "tc_gemm.cuh"

namespace tcm {

constexpr int kRows = 128, kIn = 64, kWid = 256, kLayers = 4;
constexpr int kEpiWarps = 16;  // shared by the two chains
constexpr int kThreads = 32 * (2 + kEpiWarps);  // the training kernels: producer, MMA issuer, epilogues
// inference: the issuing warps and two idle ones are a warpgroup of their own, whose registers go to the
// epilogues (setmaxnreg): launched with 96 per thread, 32 x 4 + 112 x 16 = 96 x 20 warps' worth
constexpr int kCtlWarps = 4, kCtlRegs = 32, kEpiRegs = 112, kLaunchRegs = 96;
constexpr int kInferThreads = 32 * (kCtlWarps + kEpiWarps);
static_assert(kCtlWarps * kCtlRegs + kEpiWarps * kEpiRegs <= (kCtlWarps + kEpiWarps) * kLaunchRegs, "register split");
constexpr int kChunkA = kRows * 128;  // one 128-byte-wide K chunk of an activation tile
constexpr int kChunkW = kWid * 128;   // one 128-byte-wide K chunk of a weight matrix

// Barriers and words that a CTA's roles share, behind the ring in dynamic shared memory.
template <int STAGES>
struct Control {
    uint64_t w_full[STAGES], w_empty[STAGES];
    uint64_t x_full[2], act_free[2], acc_full[2], act_ready[2], head_bar[2], drain;
    uint32_t tmem_base;
    int abort_flag;
};
constexpr int kControlBytes = 256;
static_assert(sizeof(Control<5>) <= kControlBytes, "control block");

template <bool FP8>
struct Cfg {
    static constexpr int act_bytes = FP8 ? kRows * kWid : kRows * kWid * 2;  // >= the BF16 input tile
    static constexpr int stages = FP8 ? 5 : 3;
    static constexpr int smem = 1024 + 2 * act_bytes + stages * kChunkW + kControlBytes;
    // 128-byte K chunks per layer: layer 1 reads kIn BF16 inputs
    __host__ __device__ static constexpr int chunks(int l) { return l == 0 ? kIn * 2 / 128 : (FP8 ? 2 : 4); }
};
static_assert(Cfg<false>::smem <= 227 * 1024 && Cfg<true>::smem <= 227 * 1024, "shared memory");
static_assert(kIn % 64 == 0 && kIn <= kWid, "input rows are whole 128-byte K chunks");

struct Args {
    int n;                  // feature rows
    int members;
    long long units;        // ceil(n / 128) * members (< 2^28)
    const float* master;    // FP32 parameters, member stride P
    long long P;
    long long off_b[kLayers];
    long long off_w5, off_b5;
    const float* wscale_half;  // FP8: [members][3][256] halves of the scales of W2..W4 (one per matrix, repeated per row)
    float* pred;            // [members][pred_stride]
    long long pred_stride;  // member stride of pred
    int* status;
};

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            tc::sa(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(tc::sa(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(tc::sa(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(tc::sa(bar))
        : "memory");
}

// Bulk tensor store of one box from shared memory into the issuing thread's bulk group (all
// coordinates non-negative, x a multiple of 16 bytes).
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int x, int y, int z, int w)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(tc::sa(src)), "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}

// L2 policy of training data that is read once more after it left the L2 anyway, or not again: its
// lines are given up first. A step's activations, gelu' and gradients (8,192 rows x 5 members: 270 MB)
// pass through an L2 of 129 MB, and which of them stay decides what the backward kernels wait for.
// 14 steps, starting from 2.00 ms: H1..H3 stored with it 1.97, gelu' read with it as well 1.97, the
// weight gradients' Hprev loads too 1.94, their dZ loads too 1.90. Not kept: the head backward's loads
// of H4 and gelu'(Z4) (2.04, alone).
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int x, int y, int z, int w,
                                             uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3, %4, %5}], [%1], %6;\n" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(tc::sa(src)), "r"(x), "r"(y), "r"(z), "r"(w), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar,
                                            uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
        "[%1, {%2, %3, %4}], [%5], %6;\n" ::"r"(tc::sa(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(tc::sa(bar)), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }

// The thread's committed bulk stores have read their shared-memory sources.
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }

// The thread's committed bulk stores are complete.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ void named_barrier(int id, int threads)
{
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::sa(b)) : "memory");
}

// Instruction descriptor: kind::f8f6f4, E4M3 A and B, FP32 D, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_e4m3(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Up to 16 polls of a barrier's phase, in few instructions.
__device__ __forceinline__ bool poll16(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .u32 n;\n mov.u32 n, 16;\n"
        "POLL:\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n @p bra DONE;\n"
        " sub.u32 n, n, 1;\n setp.ne.u32 q, n, 0;\n @q bra POLL;\n"
        "DONE:\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait that also gives up when another role has aborted. TIGHT polls up to 16 times between
// looks at the abort flag: the waiting warps notice a phase sooner, but take more issue slots from the
// others. It pays where the chains wait on each other's MMAs (BF16 inference: 1.82 ms per 2^20 rows x 5
// members against 1.86 without the register split), not where the epilogues set the pace (E4M3: 0.192
// against 0.186 ms per 100,003 rows; 14 training steps: 2.35 against 2.23 ms).
template <bool TIGHT = false>
__device__ __forceinline__ bool wait_bar(uint64_t* b, uint32_t parity, int* status, volatile int* abort_flag)
{
    constexpr int kPolls = TIGHT ? 16 : 1;
    const uint32_t bar = tc::sa(b);
    if (TIGHT && poll16(bar, parity)) return true;
    for (int i = 0; i < (int)(tc::kSpin / kPolls); ++i) {
        if (TIGHT ? poll16(bar, parity) : tc::mbar_try(b, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicOr(status, 2);
    return false;
}

template <int N>
__device__ __forceinline__ void reg_alloc()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_dealloc()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(N));
}

// One lane of a converged warp (the same one each time).
__device__ __forceinline__ bool elect_one()
{
    uint32_t e;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
    return e != 0;
}

// wait_bar for a whole warp: true on every lane or on none, so that the warp stays together for
// the collective loads and stores that follow.
template <bool TIGHT = false>
__device__ __forceinline__ bool wait_bar_warp(uint64_t* b, uint32_t parity, int* status, volatile int* abort_flag)
{
    return __all_sync(0xffffffffu, wait_bar<TIGHT>(b, parity, status, abort_flag));
}

// Byte offset of 16-byte unit j (0..7) of row r in a 128-row, 128-byte-wide K chunk
// laid out as TMA writes it with 128-byte swizzle (8-row groups of 1024 bytes).
__device__ __forceinline__ uint32_t swz(int r, int j) { return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((j ^ (r & 7)) << 4)); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t pack_e4m3(float a, float b, float c, float d)
{
    const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
    const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3);
    return lo | (hi << 16);
}

__device__ __forceinline__ void st_shared_v4(uint8_t* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(tc::sa(p)), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

// 16 parameters (biases or head weights, read again by every unit): kept in L1 with priority.
__device__ __forceinline__ void ld16(const float* p, float (&x)[16])
{
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        float4 q;
        asm volatile("ld.global.nc.L1::evict_last.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                     : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w)
                     : "l"(p + i));
        x[i] = q.x;
        x[i + 1] = q.y;
        x[i + 2] = q.z;
        x[i + 3] = q.w;
    }
}

using f32x2::fma2;
using f32x2::mul2;

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// 256-bit global store of eight 32-bit words (address 32-byte aligned), not kept in L1; ONCE: with the
// policy of policy_evict_first().
template <bool ONCE = false>
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t (&w)[8])
{
    if (ONCE)
        asm volatile("st.global.L1::no_allocate.L2::evict_first.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p),
                     "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
    else
        asm volatile("st.global.L1::no_allocate.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "r"(w[0]),
                     "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
}

// 256-bit global load of eight 32-bit words (address 32-byte aligned; data not written by this kernel),
// which are not read again.
__device__ __forceinline__ void ld_global_v8u(const void* p, uint32_t (&x)[8])
{
    asm volatile("ld.global.nc.L1::no_allocate.L2::evict_first.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7])
                 : "l"(p));
}

// 16 consecutive accumulator columns of this thread's TMEM lane (row), then the wait.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Waits for this thread's outstanding TMEM loads; the loaded registers pass through, so that no
// use of them moves above the wait.
template <int N>
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[N])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}

// Starts the load of eight consecutive accumulator columns of this thread's TMEM lane (row).
__device__ __forceinline__ void tmem_ld8_start(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Starts the load of 16 accumulator columns of 16 TMEM lanes as two 8-column fragments: registers
// 4 c .. 4 c + 3 hold columns 8 c + 2 (lane & 3) + {0, 1} of rows lane / 4 and lane / 4 + 8.
__device__ __forceinline__ void tmem_ldfrag_start(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Four 8 x 8 matrices of 16-bit values in fragment layout to shared memory; lane i gives the
// address of row i & 7 of matrix i / 8 (16 bytes).
__device__ __forceinline__ void st_matrix_x4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(a), "r"(b),
                 "r"(c), "r"(d)
                 : "memory");
}

// Two parameters (a fragment's column pair), kept in L1 with priority.
__device__ __forceinline__ float2 ld2(const float* p)
{
    float2 q;
    asm volatile("ld.global.nc.L1::evict_last.v2.f32 {%0, %1}, [%2];\n" : "=f"(q.x), "=f"(q.y) : "l"(p));
    return q;
}

__device__ __forceinline__ void ld8(const float* p, float (&x)[8])
{
#pragma unroll
    for (int i = 0; i < 8; i += 4)
        asm volatile("ld.global.nc.L1::evict_last.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                     : "=f"(x[i]), "=f"(x[i + 1]), "=f"(x[i + 2]), "=f"(x[i + 3])
                     : "l"(p + i));
}

// 2 gelu(z) = z (1 + tanh u), u = z (K C z^2 + K), on a pair, in FP32: one multi-function-unit tanh
// per element, the rest packed FP32x2 operations (half the instructions of the scalar form).
__device__ __forceinline__ float2 gelu_tanh(float2 z)
{
    const float2 u = mul2(z, fma2(f2(mlp::kGeluK * mlp::kGeluC), mul2(z, z), f2(mlp::kGeluK)));
    return make_float2(mlp::tanh_hw(u.x), mlp::tanh_hw(u.y));
}

__device__ __forceinline__ float2 as_pair(uint32_t a, uint32_t b) { return make_float2(__uint_as_float(a), __uint_as_float(b)); }

// ---- epilogues of 128 accumulator columns of a warp's 32 rows ----
//
// Each runs as a software pipeline over blocks of eight values per thread: a block's tanh are issued
// (`pre`) before the block before it is finished and stored (`post`), and the next block's accumulator
// columns and parameters are requested before that.

// Hidden layers of BF16 inference: fragments of 16 rows x 8 columns (tmem_ldfrag_start), so that a
// parameter load serves four rows, and the pairs go to act (BF16 of 2 h) with stmatrix. taddr:
// accumulator of the warp's rows and columns; bias: its columns' biases; act: its first K chunk.
__device__ __forceinline__ void epi_frag(uint32_t taddr, const float* bias, uint8_t* act, int q, int lane, float acc_mul,
                                         const float2 (&b0)[2])
{
    const float* bp = bias + 2 * (lane & 3);
    // stmatrix row of this lane: row (lane & 7) + 8 (bit 3), column group + bit 4
    const uint32_t dst = tc::sa(act) + (uint32_t)((q * 4 + ((lane >> 3) & 1)) * 1024 + (lane & 7) * 128);
    const uint32_t unit = (uint32_t)(((lane >> 4) ^ (lane & 7)) << 4);
    uint32_t v[2][8];
    float2 z[2][4], t[2][4], bb[2][2] = {{b0[0], b0[1]}, {b0[0], b0[1]}};
    // block b: columns 16 (b / 2).., rows 16 (b % 2)..
    auto start = [&](int b) { tmem_ldfrag_start(taddr + ((uint32_t)(16 * (b & 1)) << 16) + 16 * (b >> 1), v[b & 1]); };
    auto pre = [&](int b) {
        const int p = b & 1, cg = b >> 1;
        tmem_wait_ld(v[p]);
        if (b < 15) start(b + 1);
        if (p == 0 && cg < 7) {
#pragma unroll
            for (int c = 0; c < 2; ++c) bb[(cg + 1) & 1][c] = ld2(bp + 16 * (cg + 1) + 8 * c);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // (column group i / 2, row half i % 2)
            z[p][i] = fma2(as_pair(v[p][2 * i], v[p][2 * i + 1]), f2(acc_mul), bb[cg & 1][i >> 1]);
            t[p][i] = gelu_tanh(z[p][i]);
        }
    };
    auto post = [&](int b) {
        const int p = b & 1, cg = b >> 1;
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 h = fma2(z[p][i], t[p][i], z[p][i]);
            w[i] = pack_bf16(h.x, h.y);
        }
        st_matrix_x4(dst + (uint32_t)((cg >> 2) * kChunkA + p * 2048) + (unit ^ (uint32_t)((2 * (cg & 3)) << 4)), w[0],
                     w[1], w[2], w[3]);
    };
    start(0);
    pre(0);
#pragma unroll
    for (int b = 0; b < 16; ++b) {
        if (b < 15) pre(b + 1);
        post(b);
    }
}

// Thread = row: the head (either variant), and the hidden layers of E4M3 inference (a 16-byte unit of
// codes of 2 h per 16 columns). b0, w0: the first eight biases and head weights. act: the chain's
// buffer; r: row in the tile; c_beg: first column. yh: the head's sums over each 64 columns.
template <bool HEAD>
__device__ __forceinline__ void epi_rows(uint32_t taddr, const float* bias, const float* w5, uint8_t* act, int r, int c_beg,
                                         float mul, const float (&b0)[8], const float (&w0)[8], float (&yh)[2])
{
    uint32_t v[2][8], w[4];
    float2 z[2][4], t[2][4];
    float bb[8], ww[2][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        bb[i] = b0[i];
        if (HEAD) ww[0][i] = w0[i];
    }
    auto start = [&](int b) { tmem_ld8_start(taddr + 8 * b, v[b & 1]); };
    auto pre = [&](int b) {
        const int p = b & 1;
        tmem_wait_ld(v[p]);
        if (b < 15) start(b + 1);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            z[p][i] = fma2(as_pair(v[p][2 * i], v[p][2 * i + 1]), f2(mul), make_float2(bb[2 * i], bb[2 * i + 1]));
        if (b < 15) ld8(bias + 8 * (b + 1), bb);
        if (HEAD && b > 0) ld8(w5 + 8 * b, ww[p]);
#pragma unroll
        for (int i = 0; i < 4; ++i) t[p][i] = gelu_tanh(z[p][i]);
    };
    auto post = [&](int b) {
        const int p = b & 1;
        float2 h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            h[i] = fma2(z[p][i], t[p][i], z[p][i]);
            if (HEAD) {  // on 2 h4; the sum is halved with b5 added by the caller
                yh[b >> 3] = fmaf(ww[p][2 * i], h[i].x, yh[b >> 3]);
                yh[b >> 3] = fmaf(ww[p][2 * i + 1], h[i].y, yh[b >> 3]);
            }
        }
        if (HEAD) return;
        w[2 * p] = pack_e4m3(h[0].x, h[0].y, h[1].x, h[1].y);
        w[2 * p + 1] = pack_e4m3(h[2].x, h[2].y, h[3].x, h[3].y);
        const int col = c_beg + 8 * (b - 1);
        if (p) st_shared_v4(act + (col >> 7) * kChunkA + swz(r, (col & 127) >> 4), w[0], w[1], w[2], w[3]);
    };
    start(0);
    pre(0);
#pragma unroll
    for (int b = 0; b < 16; ++b) {
        if (b < 15) pre(b + 1);
        post(b);
    }
}

// A persistent CTA's unit of ordinal jj: tile and member (units < 2^28, so 32-bit division). Units are
// member by member, so that all CTAs work on one member at a time: its biases and head weights (5 KB)
// stay in the L1 cache that the ring leaves (28 KB), its weights in L2; tile by tile the members'
// 25 KB did not fit (63 % L1 hits).
struct Unit {
    int tile, mem;
};
__device__ __forceinline__ Unit unit_at(int jj, int tiles)
{
    const unsigned u = blockIdx.x + (unsigned)jj * gridDim.x;
    const unsigned m = u / (unsigned)tiles;
    return {(int)(u - m * (unsigned)tiles), (int)m};
}

// grid: min(SMs, units) persistent CTAs; CTA b runs units b, b + gridDim.x, ...;
// its j-th unit goes to chain j % 2. Unit u = (tile u % tiles, member u / tiles).
// 96 registers per thread at launch: five warps on each of the SM's four sub-partitions of 16,384
// registers (5 x 32 x 96 = 15,360; at 104 the launch does not fit).
template <bool FP8>
__global__ void __maxnreg__(kLaunchRegs) mlp_infer_kernel(const __grid_constant__ CUtensorMap tx,
                                                 const __grid_constant__ CUtensorMap tw1,
                                                 const __grid_constant__ CUtensorMap tw,
                                                 const __grid_constant__ Args g)
{
    using C = Cfg<FP8>;
    extern __shared__ uint8_t smem_raw[];

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ring = smem + 2 * C::act_bytes;
    Control<C::stages>& ctl = *reinterpret_cast<Control<C::stages>*>(ring + C::stages * kChunkW);
    // the warp number through a shuffle, so that the roles' branches and the MMA issuer's descriptor
    // arithmetic compile as warp-uniform
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int units = (int)g.units, tiles = units / g.members;
    const int my_units = units > (int)blockIdx.x ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    volatile int* abort_v = &ctl.abort_flag;

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
            tc::mbar_init(&ctl.act_ready[s], kEpiWarps / 2);
            tc::mbar_init(&ctl.head_bar[s], kEpiWarps / 4);
        }
        tc::mbar_init(&ctl.drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        ctl.abort_flag = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = ctl.tmem_base;

    if (warp < kCtlWarps) {
        reg_dealloc<kCtlRegs>();
        if (warp == 0) {
            // ---- producer: per unit pair, layer by layer, chain by chain (the MMA order) ----
            if (lane == 0) {
                int st = 0, issued = 0;      // ring stage of the next weight chunk; stages filled at least once
                uint32_t wph = 1;            // parity of w_empty for it (the first pass over the ring does not wait)
                int x_last[2] = {-1, -1};    // last unit whose input rows were requested, per chain
                bool ok = true;
                for (int j = 0; j < my_units && ok; j += 2) {
                    const Unit un[2] = {unit_at(j, tiles), unit_at(j + 1, tiles)};
                    const int ns = min(2, my_units - j);
                    for (int l = 0; l < kLayers && ok; ++l) {
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            if (s >= ns || !ok) break;
                            if (l == 0) {
                                // the chain's buffer is free once the unit two before finished its MMAs
                                if (j >= 2 && !(ok = wait_bar<!FP8>(&ctl.act_free[s], (uint32_t)(((j - 2) >> 1) & 1), g.status,
                                                              abort_v)))
                                    break;
                                uint8_t* act = smem + s * C::act_bytes;
                                tc::mbar_expect_tx(&ctl.x_full[s], C::chunks(0) * kChunkA);
                                for (int c = 0; c < C::chunks(0); ++c)
                                    tma_load_2d(act + c * kChunkA, &tx, c * 16, un[s].tile * kRows, &ctl.x_full[s]);
                                x_last[s] = j + s;
                            }
                            for (int c = 0; c < C::chunks(l); ++c) {
                                if (!(ok = wait_bar<!FP8>(&ctl.w_empty[st], wph, g.status, abort_v))) break;
                                tc::mbar_expect_tx(&ctl.w_full[st], kChunkW);
                                // maps address 8-byte elements: 16 per 128-byte K chunk
                                if (l == 0)
                                    tc::tma_load_3d(ring + st * kChunkW, &tw1, c * 16, 0, un[s].mem, &ctl.w_full[st]);
                                else
                                    tma_load_4d(ring + st * kChunkW, &tw, c * 16, 0, l - 1, un[s].mem, &ctl.w_full[st]);
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
            for (int j = 0; j < my_units && ok; j += 2) {
                const int ns = min(2, my_units - j);
                for (int l = 0; l < kLayers && ok; ++l) {
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        if (s >= ns || !ok) break;
                        if (l == 0 && !(ok = wait_bar_warp<!FP8>(&ctl.x_full[s], (uint32_t)((j >> 1) & 1), g.status, abort_v)))
                            break;
                        if (!(ok = wait_bar_warp<!FP8>(&ctl.w_full[st], wph, g.status, abort_v))) break;
                        // the epilogue of the chain's previous layer (ordinal 4 (j / 2) + l - 1) has
                        // written act and drained acc
                        if ((j | l) != 0 &&
                            !(ok = wait_bar_warp<!FP8>(&ctl.act_ready[s], (uint32_t)((l - 1) & 1), g.status, abort_v)))
                            break;
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        const uint8_t* act = smem + s * C::act_bytes;
                        const uint32_t d = tmem + (uint32_t)(s * kWid);
                        const bool f8 = FP8 && l > 0;
                        const uint64_t a = tc::sdesc(act);  // addresses in the descriptors count 16-byte units
#pragma unroll
                        for (int c = 0; c < C::chunks(1); ++c) {
                            if (c >= C::chunks(0) && l == 0) break;
                            if (c > 0) {
                                if (!(ok = wait_bar_warp<!FP8>(&ctl.w_full[st], wph, g.status, abort_v))) break;
                                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                            }
                            const uint64_t b = b_ring + (uint64_t)(st * (kChunkW >> 4));
                            if (leader) {
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk) {
                                    if (f8)
                                        mma_e4m3(d, a + c * (kChunkA >> 4) + kk * 2, b + kk * 2, idesc_e4m3(kRows, kWid), (c | kk) != 0);
                                    else
                                        tc::mma_bf16(d, a + c * (kChunkA >> 4) + kk * 2, b + kk * 2, tc::idesc_bf16(kRows, kWid), (c | kk) != 0);
                                }
                                tc::mma_commit(&ctl.w_empty[st]);
                            }
                            if (++st == C::stages) {
                                st = 0;
                                wph ^= 1;
                            }
                        }
                        if (!ok) break;
                        if (leader) {
                            tc::mma_commit(&ctl.acc_full[s]);
                            if (l == kLayers - 1) tc::mma_commit(&ctl.act_free[s]);
                        }
                        __syncwarp();
                    }
                }
            }
            if (leader) {
                tc::mma_commit(&ctl.drain);  // arrives when every MMA issued above has completed
                tc::mbar_wait(&ctl.drain, 0, g.status);
            }
            __syncwarp();
        }
    } else {
        reg_alloc<kEpiRegs>();
        // ---- epilogue: eight warps per chain; warp = (TMEM lane quarter q, column half ch) ----
        const int s = (warp - kCtlWarps) >> 3, q = warp & 3, ch = ((warp - kCtlWarps) >> 2) & 1;
        const int r = q * 32 + lane;  // row in the tile where thread = accumulator row
        const int c_beg = ch * (kWid / 2);
        uint8_t* act = smem + s * C::act_bytes;
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(s * kWid + c_beg);
        bool ok = true;
        for (int j = s; j < my_units && ok; j += 2) {
            const Unit un = unit_at(j, tiles);
            const int tile = un.tile, mem = un.mem;
            const float* prm = g.master + mem * g.P;
            for (int l = 0; l < kLayers && ok; ++l) {
                const float* bias = prm + g.off_b[l] + c_beg;
                // layers 2-4 read 2 h (see the header), so their accumulator is halved here
                const float acc_mul = l > 0 ? 0.5f : 1.0f;
                const uint32_t acc_ph = (uint32_t)(l & 1);  // of ordinal 4 (j / 2) + l
                // E4M3 layers: the accumulator times half the matrix's weight scale
                const float mul =
                    FP8 && l > 0 ? __ldg(g.wscale_half + ((long long)mem * 3 + (l - 1)) * kWid) : acc_mul;
                const int row = tile * kRows + r;
                float yh[2] = {0.0f, 0.0f};  // head sums of the warp's two column quarters
                if (l == kLayers - 1) {
                    const float* w5 = prm + g.off_w5 + c_beg;
                    float b0[8], w0[8];
                    ld8(bias, b0);
                    ld8(w5, w0);
                    if (!(ok = wait_bar_warp<!FP8>(&ctl.acc_full[s], acc_ph, g.status, abort_v))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    epi_rows<true>(taddr, bias, w5, act, r, c_beg, mul, b0, w0, yh);
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    // the upper half's head sums for the lower half, in the chain's second K chunk: its
                    // MMAs are done, and the next unit writes it only after the lower half has arrived
                    // on act_ready below
                    float* part = reinterpret_cast<float*>(act + kChunkA);
                    if (ch) {
                        part[r] = yh[0];
                        part[kRows + r] = yh[1];
                        __syncwarp();
                        if (lane == 0) {
                            mbar_arrive(&ctl.head_bar[s]);
                            mbar_arrive(&ctl.act_ready[s]);
                        }
                    } else {
                        if (!(ok = wait_bar_warp<!FP8>(&ctl.head_bar[s], (uint32_t)((j >> 1) & 1), g.status, abort_v))) break;
                        const float sum = ((yh[0] + yh[1]) + part[r]) + part[kRows + r];
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ctl.act_ready[s]);
                        if (row < g.n)
                            g.pred[(long long)mem * g.pred_stride + row] = fmaf(sum, 0.5f, prm[g.off_b5]);
                    }
                    continue;
                }
                if constexpr (!FP8) {
                    const float2 b0[2] = {ld2(bias + 2 * (lane & 3)), ld2(bias + 2 * (lane & 3) + 8)};
                    if (!(ok = wait_bar_warp<!FP8>(&ctl.acc_full[s], acc_ph, g.status, abort_v))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    epi_frag(taddr, bias, act + 2 * ch * kChunkA, q, lane, acc_mul, b0);
                } else {
                    float b0[8];
                    ld8(bias, b0);
                    if (!(ok = wait_bar_warp<!FP8>(&ctl.acc_full[s], acc_ph, g.status, abort_v))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    epi_rows<false>(taddr, bias, nullptr, act, r, c_beg, mul, b0, b0, yh);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl.act_ready[s]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
}

}  // namespace tcm
