// Chunked tensor-core WKV-6 prefill for sm_100a (tcgen05 + TMEM + TMA).
//
// One CTA per (sequence, head) walks the sequence in chunks of L = 64 tokens.  With the
// in-chunk inclusive cumulative log2-decay a_t = sum_{s<=t} log2 w_s (a_0 = 0, fp32, restarted
// every chunk) and the chunk's start state S_0, the recurrence re-associates exactly to
//   y_t  = (r_t * 2^{a_{t-1}}) . S_0 + sum_{i<t} P[t,i] v_i + (sum_c r_t[c] u[c] k_t[c]) v_t
//   P[t,i] = sum_c (r_t[c] 2^{a_{t-1}[c]}) (k_i[c] 2^{-a_i[c]})
//   S_L  = diag(2^{a_L}) ( S_0 + sum_i (k_i * 2^{-a_i})^T v_i )
// so a chunk is four 64x64x64 bf16 contractions (fp32 accumulate) around an fp32 elementwise
// phase.  The contractions are tcgen05.mma instructions issued by elected lanes of two warps, with operands in
// 128-byte-swizzled shared memory tiles (the layout TMA delivers) and accumulators in tensor
// memory; score, state-increment and output accumulators are double buffered there so the
// tensor pipe runs one chunk ahead of the warps that read them back.
// The single in-chunk reference point is safe while no channel decays by more than 2^-96 inside
// one chunk (always true for w >= 0.36; the benchmark's decays are >= 0.69); a chunk that
// violates it is processed token by token in fp32 instead, so any finite or infinite decay
// logit gives the exact-recurrence result.
//
// Warp roles (992 threads), pipelined across chunks through mbarriers:
//   warp 0        TMA producer: {x,r,k,v} tiles of a chunk into one stage of a 5-stage ring
//   warp 1        tensor-memory allocation; an elected lane issues P = R^ K^^T and dS = K^^T V
//   warp 2        an elected lane issues Y = R^ S_0 + P' V (one accumulator)
//   warps 3-6     state: S <- diag(2^{a_L}) (S + dS) in fp32 registers for the whole sequence;
//                 publishes a bf16 copy of every chunk-start state as an MMA operand; for a chunk on
//                 the token-by-token path it parks the fp32 state in shared memory instead
//   warps 7-10    scores: P from tensor memory -> P' = tril(P,-1) + diag(bonus) -> bf16 operand tile
//   warps 11-14   output: Y from tensor memory -> bf16 -> TMA store (each warp its own 16 rows);
//                 runs the token-by-token path (16 value channels per warp) when a chunk needs it
//   warps 15-30   elementwise, two sets of eight warps taking alternate chunks: decay and
//                 cumulative sum (phase A), then in place R^ = r 2^{a_{t-1}}, K^ = k 2^{-a_t}
//                 (phase B); chunk decay 2^{a_L}, bonus coefficients, safety vote.  A lane owns
//                 4 tokens x 4 channels (64-bit shared-memory accesses, packed fp32x2 arithmetic)
// A warp reads the tensor-memory lanes of its own sub-partition (warp index mod 4), which hold
// accumulator rows 16*(warp mod 4) .. +15 of a 64-row tile.
// Every wait is bounded: on expiry the kernel raises a status flag and all roles leave.
//
// Three template parameters select variants of the same pipeline: SUMMARY (the first pass of a call
// that splits its sequences into segments: state only, no r / scores / outputs; see Params), C2
// (the Finch-C2 form: keys times one minus their decay, no bonus, optional per-token vector added to
// the output) and PERSIST (calls with more units than SMs: one CTA per SM walks a stream of units,
// the producer leaving a descriptor per chunk and two end markers that every role hands on, so that
// the pipeline is filled and drained once per CTA instead of once per unit; PERSIST = 2 also cuts units
// between neighbouring CTAs, so that every CTA gets the same number of chunks: see Params::bal_chunks).
#pragma once
#include <atomic>
#include <chrono>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "device_info.cuh"
#include "gf_wkv6.h"

namespace gf {

__device__ int g_dev_status = 0;

inline cudaError_t read_and_clear_device_status(int* flag)
{
    cudaError_t e = cudaMemcpyFromSymbol(flag, g_dev_status, sizeof(int));
    if (e != cudaSuccess) return e;
    if (*flag) {
        int z = 0;
        e = cudaMemcpyToSymbol(g_dev_status, &z, sizeof(int));
    }
    return e;
}

namespace ck {

constexpr int L = 64;                  // tokens per chunk
constexpr int TILE = 64 * 64 * 2;      // one bf16 [64 x 64] tile
constexpr int NS = 5;                  // {x,r,k,v} ring depth
constexpr int NSB = 2;                 // bf16 chunk-start state operand tiles (by chunk parity)
constexpr int NPP = 2;                 // bf16 masked-score operand tiles (by chunk parity)
constexpr int NSIDE = 8;               // ring of per-chunk side vectors (chunk decay, bonus, safety flag): deeper than
                                       // every consumer's lag behind the elementwise warps, so it needs no release
constexpr int NTOT = 4;                // per-warp decay-total buffers (two per elementwise set)
constexpr int N_EW = 8;                // elementwise warps per set
constexpr int N_ESET = 2;              // elementwise sets (alternate chunks)
// The ring is waited on by two sets that take alternate chunks, and its depth is odd: a stage belongs to either set in turn.  A
// wait names a phase by its parity alone, so a set has to meet every phase of the barriers it waits on.  Hence a "full" barrier
// per set and stage, which only that set waits on.  (One barrier per stage would let a set through to chunk c while the copy of
// chunk c - NS, which had the stage before, is still landing.)  Chunk c takes stage 3 c mod 5, so that a set's next chunk takes
// the next stage and its phase bit flips where the stage wraps; set 1 begins at stage 3, so its barriers of the stages before
// that start one phase ahead.
constexpr int STAGE_STEP = 3;
static_assert(NS == 5 && N_ESET == 2 && STAGE_STEP * N_ESET % NS == 1, "the stages of a set's chunks follow one another");
__device__ __forceinline__ void next_stage(int& s, int& ph)      // for the roles that take every chunk: the phase flips every NS chunks
{
    s += STAGE_STEP;
    if (s >= NS) s -= NS;
    if (s == 0) ph ^= 1;
}
constexpr int N_GW = 4;                // warps per tensor-memory reader group (one per sub-partition)
constexpr int WARP_MMA_F = 1;          // issues P = R^ K^^T and dS = K^^T V; owns the tensor-memory allocation
constexpr int WARP_MMA_B = 2;          // issues Y = R^ S_0 + P' V
constexpr int WARP_S0 = 3;             // state warps
constexpr int WARP_P0 = WARP_S0 + N_GW;   // score warps
constexpr int WARP_Y0 = WARP_P0 + N_GW;   // output warps
constexpr int WARP_E0 = WARP_Y0 + N_GW;   // elementwise warps
constexpr int THREADS = 32 * (WARP_E0 + N_ESET * N_EW);
constexpr float A2_MAX = 96.f;         // largest in-chunk |cumulative log2 decay| on the tensor-core path
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LOG2_LOG2E = 0.5287663729448977f;
constexpr uint32_t WAIT_LIMIT_US = 2000000u;                   // default limit of a device-side wait: 2 s
constexpr uint32_t TRY_WAIT_HINT_NS = 20000;                  // a waiting thread may be suspended this long per try

// tensor memory: 64 fp32 columns per 64x64 accumulator, two buffers each
constexpr int TM_COLS = 512;          // (384 are used; the allocation is a power of two)
constexpr int TM_P = 0, TM_DS = 128, TM_Y = 256;

// shared memory map (offsets from a 1024-byte aligned base)
constexpr int STAGE = 4 * TILE;                            // one ring stage: x, r -> R^, k -> K^, v
constexpr int OFF_RING = 0;                                // [NS][STAGE]
constexpr int OFF_SB = OFF_RING + NS * STAGE;              // [NSB][TILE]          bf16 chunk-start state [c][j]
constexpr int OFF_PP = OFF_SB + NSB * TILE;                // [NPP][TILE]          bf16 masked scores [t][i]
constexpr int OFF_Y = OFF_PP + NPP * TILE;                 // [N_GW][16 rows x 128 B] y staging, one slab per warp
constexpr int OFF_U2 = OFF_Y + N_GW * 2048;                // [N_GW][16 rows x 128 B] second-value slabs (Finch-C2 form)
constexpr int OFF_TOT = OFF_U2 + N_GW * 2048;              // [NTOT][N_EW][64] float
constexpr int OFF_DL = OFF_TOT + NTOT * N_EW * 64 * 4;     // [NSIDE][64] float    2^{a_L}
constexpr int OFF_DU = OFF_DL + NSIDE * 64 * 4;            // [NSIDE][64] float    bonus coefficient per token
constexpr int OFF_SAFE = OFF_DU + NSIDE * 64 * 4;          // [NSIDE] int
constexpr int OFF_ABORT = OFF_SAFE + NSIDE * 4;            // int
constexpr int OFF_TMEM = OFF_ABORT + 8;                    // uint32: tensor-memory base address
constexpr int OFF_BAR = OFF_ABORT + 16;                    // mbarriers (8 bytes each)
enum {
    BAR_FULL_RKV = 0,                    // copies of a chunk landed (by set and stage)
    BAR_EMPTY_RKV = BAR_FULL_RKV + N_ESET * NS,
    BAR_RK_READY = BAR_EMPTY_RKV + NS,
    BAR_S_READY = BAR_RK_READY + NS,     // bf16 state operand tile written            (by chunk parity)
    BAR_PP_READY = BAR_S_READY + 2,      // masked-score operand tile written
    BAR_F_FULL = BAR_PP_READY + 2,       // P and dS accumulators complete
    BAR_F_EMPTY = BAR_F_FULL + 2,        // ... and read back by the state and score warps
    BAR_B_DONE = BAR_F_EMPTY + 2,        // Y accumulator complete; state / score operand tiles free again
    BAR_Y_EMPTY = BAR_B_DONE + 2,        // ... and read back by the output warps
    BAR_ESYNC = BAR_Y_EMPTY + 2,         // one per elementwise set
    BAR_SSYNC = BAR_ESYNC + 2,           // token-by-token path only: state-warp rendezvous after the fp32 copy is re-read,
    BAR_SPRE = BAR_SSYNC + 1,            //   and before it is written,
    BAR_FB_READY = BAR_SPRE + 1,         //   fp32 state copy in place for the output warps,
    BAR_FB_DONE = BAR_FB_READY + 1,      //   and advanced by them over the chunk
    BAR_U2 = BAR_FB_DONE + 1,            // Finch-C2 form: per output warp and slab, its second-value rows have landed
    BAR_COUNT = BAR_U2 + 2 * N_GW
};
// persistent launches: one descriptor per chunk of the CTA's chunk stream
// {first row, valid tokens | flags | head << 16, unit, chunks left in the unit}
constexpr int STREAM_MAX_HEADS = 65536;                          // (a descriptor's upper 16 bits; more heads: one CTA per unit)
constexpr int OFF_DESC = (OFF_BAR + BAR_COUNT * 8 + 15) & ~15;   // [NSIDE] int4
// flags beside the valid-token count (low byte): first chunk of a unit (or piece of one), no chunk, piece that continues
// a unit another CTA began, last chunk of a piece
constexpr int DESC_FIRST = 0x100, DESC_END = 0x200, DESC_CONT = 0x400, DESC_LAST = 0x800;
constexpr int DESC_TAG = 0x1000;                                 // (balanced launches) parity of the ring's turn: (chunk / NSIDE) & 1
constexpr int OFF_MARK = OFF_DESC + NSIDE * 16;                  // int: the segment's state became non-finite (Params::trail)
constexpr int SMEM_BYTES = OFF_MARK + 16;
constexpr int SMEM_ALLOC = SMEM_BYTES + 1024;              // slack for manual 1024-byte alignment
static_assert(SMEM_ALLOC <= 232448, "shared memory budget of one sm_100 CTA");

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrival by the lanes whose predicate holds, as one predicated instruction (no divergent branch).
__device__ __forceinline__ void mbar_arrive_if(uint32_t bar, bool pred)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
        ::"r"(bar), "r"((uint32_t)pred) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ float ldsf(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void stsf(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void stsf_if(uint32_t a, float v, bool pred)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(a), "f"(v), "r"((uint32_t)pred) : "memory");
}
__device__ __forceinline__ float4 ldsf4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void stsf4(uint32_t a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void stsf4_if(uint32_t a, float4 v, bool pred)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n\t}"
                 ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((uint32_t)pred) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(TRY_WAIT_HINT_NS) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait.  Returns false if the CTA is aborting or the wait ran out of time (the
// status flag is then raised and the CTA-wide abort flag set so every role leaves).  The limit, in
// microseconds, is the 32-bit word that follows the abort word in shared memory.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint32_t abort_flag, bool poll_abort)
{
    const unsigned long long t0 = globaltimer();
    const unsigned long long limit_ns = 1000ull * lds32(abort_flag + 4);
    for (;;) {
        for (int it = 0; it < 64; ++it)
            if (mbar_try_wait(bar, parity)) return true;
        if (poll_abort && lds32(abort_flag)) return false;
        if (globaltimer() - t0 > limit_ns) break;
        __nanosleep(64);
    }
    sts32(abort_flag, 1u);
    atomicExch(&g_dev_status, 1);
    return false;
}
// abort_flag: shared-memory address of the CTA-wide abort word (followed by the wait limit)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t abort_flag, bool poll_abort = true)
{
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, poll_abort);
}

// Bounded wait for the tag of a chunk descriptor in shared memory; false as above.
__device__ __noinline__ bool desc_wait(uint32_t meta_addr, uint32_t tag, uint32_t abort_flag)
{
    const unsigned long long t0 = globaltimer();
    const unsigned long long limit_ns = 1000ull * lds32(abort_flag + 4);
    for (;;) {
        for (int it = 0; it < 64; ++it) {
            uint32_t m;
            asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(m) : "r"(meta_addr) : "memory");
            if ((m & (uint32_t)DESC_TAG) == tag) return true;
        }
        if (lds32(abort_flag)) return false;
        if (globaltimer() - t0 > limit_ns) break;
        __nanosleep(64);
    }
    sts32(abort_flag, 1u);
    atomicExch(&g_dev_status, 1);
    return false;
}
// Bounded wait of one lane for a word another CTA writes (with release semantics); false as above.
__device__ __noinline__ bool word_wait(const unsigned long long* w, unsigned long long value, uint32_t abort_flag)
{
    const unsigned long long t0 = globaltimer();
    const unsigned long long limit_ns = 1000ull * lds32(abort_flag + 4);
    for (;;) {
        for (int it = 0; it < 64; ++it) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(w) : "memory");
            if (v == value) return true;
        }
        if (lds32(abort_flag)) return false;
        if (globaltimer() - t0 > limit_ns) break;
        __nanosleep(64);
    }
    sts32(abort_flag, 1u);
    atomicExch(&g_dev_status, 1);
    return false;
}

// Warp-uniform form: every lane of a converged warp waits and all get the same answer, so the
// caller's control flow stays uniform (the compiler can then keep addresses in uniform registers).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, uint32_t abort_flag, bool poll_abort = true)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, poll_abort));
}
// True on exactly one lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(tm), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
// Asks the TMA unit to bring a tile into L2 (no shared-memory destination, no completion to wait for).
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* tm, int c0, int c1)
{
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tm), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* tm, int c0, int c1, uint32_t src)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(tm), "r"(c0), "r"(c1), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
template <int N> __device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- tensor memory and tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols)      // one full warp
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)       // the allocating warp
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The mbarrier receives one arrival once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], 64 x 64 x 16, bf16 operands, fp32 accumulate
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Shared-memory matrix descriptor of a 128-byte-swizzled [64 rows x 128 B] bf16 tile (1024-byte
// aligned): 8-row groups 1024 bytes apart.  K-major use (contraction index along the 128-byte
// row): step 32 bytes per 16 contraction indices.  MN-major use (contraction index = row): step
// 2048 bytes (16 rows) per 16 contraction indices.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3ffffu) >> 4)      // start address
         | (uint64_t)1 << 16                        // leading byte offset (unused by these shapes)
         | (uint64_t)(1024 >> 4) << 32              // stride byte offset: 8 rows
         | (uint64_t)1 << 46                        // descriptor version (sm_100)
         | (uint64_t)2 << 61;                       // 128-byte swizzle
}
// Instruction descriptor: fp32 accumulator, bf16 A and B, M = N = 64; bits 15 / 16 select the
// MN-major (transposed) form of A / B.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((64u >> 4) << 24);
constexpr uint32_t IDESC_K_K = IDESC;
constexpr uint32_t IDESC_K_MN = IDESC | (1u << 16);
constexpr uint32_t IDESC_MN_MN = IDESC | (1u << 15) | (1u << 16);

// Reads 16 rows x 32 fp32 columns of an accumulator from this warp's sub-partition and waits for
// the data: v[n][0..1] = (row g, cols 8n+2q, +1), v[n][2..3] = (row g+8, same cols) relative to the
// address, with g = lane / 4, q = lane % 4.
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, float (&v)[4][4])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(v[0][0]), "=f"(v[0][1]), "=f"(v[0][2]), "=f"(v[0][3]), "=f"(v[1][0]), "=f"(v[1][1]), "=f"(v[1][2]), "=f"(v[1][3]),
          "=f"(v[2][0]), "=f"(v[2][1]), "=f"(v[2][2]), "=f"(v[2][3]), "=f"(v[3][0]), "=f"(v[3][1]), "=f"(v[3][2]), "=f"(v[3][3])
        : "r"(taddr) : "memory");
}

// The same for 16 columns (two 8-column blocks).
__device__ __forceinline__ void tmem_ld_16x16(uint32_t taddr, float (&v)[2][4])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(v[0][0]), "=f"(v[0][1]), "=f"(v[0][2]), "=f"(v[0][3]), "=f"(v[1][0]), "=f"(v[1][1]), "=f"(v[1][2]), "=f"(v[1][3])
        : "r"(taddr) : "memory");
}

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// two-lane fp32 arithmetic on float2 values
#ifndef GF_SCALAR_F32
__device__ __forceinline__ unsigned long long pk(float2 a)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 upk(unsigned long long r)
{
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
    return upk(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
#else
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
#endif
__device__ __forceinline__ float2 ex2_2(float2 a) { return make_float2(ex2(a.x), ex2(a.y)); }
__device__ __forceinline__ uint2 lds64(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts64(uint32_t a, uint2 v)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
// the same at a compile-time byte offset from the address (folded into the instruction)
template <int OFF> __device__ __forceinline__ uint2 lds64_at(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF> __device__ __forceinline__ void sts64_at(uint32_t a, uint2 v)
{
    asm volatile("st.shared.v2.u32 [%0+%3], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y), "n"(OFF) : "memory");
}
__device__ __forceinline__ void sts128z(uint32_t a)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(0u) : "memory");
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float2 bf_pair(uint32_t w) { return make_float2(bf_lo(w), bf_hi(w)); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&p);
}
// byte offset of (row, byte-in-row) inside a 128B-swizzled [64 x 128 B] tile
__device__ __forceinline__ uint32_t swz(int row, int byte) { return (uint32_t)(row * 128 + (byte ^ ((row & 7) << 4))); }

__device__ __forceinline__ void stsm_x4(uint32_t a, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};"
                 ::"r"(a), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t a, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(a) : "memory");
}

struct Params {
    const __nv_bfloat16 *r, *k, *v, *x;   // raw pointers, used only by the token-by-token path
    __nv_bfloat16* y;
    const float* u;
    const float* state_in;
    float* state_out;
    const int32_t* cu_seqlens;             // nullptr: dense
    int T;                                 // dense sequence length
    int H;
    // Sequence split (dense calls with few (sequence, head) units): every sequence is cut into nseg
    // segments of seg_chunks chunks (the last takes the rest).  A summary launch (grid = units x
    // (nseg - 1)) leaves, per segment but the last, its decay product D[64] and the state dS[64][64] it
    // reaches from a zero start in `summaries` ([unit][segment][64 + 4096] fp32); the main launch
    // (grid = units x nseg) folds the summaries before its segment into its start state:
    // S <- diag(D) S + dS, the associative scan step across segments.  nseg = 1: no split.
    float* summaries;
    int seg_chunks;
    int nseg;
    // Finch-C2 form (the paper's Finch-C2 block): c2 != 0 multiplies every key by one minus the decay of
    // its own token and drops the bonus (u is not read); u2, if not NULL, is the per-token second-value
    // vector [rows][H*64] bf16 added to the output.
    const __nv_bfloat16* u2;
    int c2;
    // Persistent launches (more units than SMs): the grid is one CTA per SM and every CTA walks a stream
    // of units without draining its pipeline in between.  n_units = sequences x heads; `ticket`, if not
    // NULL, is a zeroed device counter from which the CTAs draw units (packed calls, whose units differ
    // in length); NULL: unit = blockIdx.x + k gridDim.x (equal lengths).
    int n_units;
    unsigned int* ticket;
    // With a ticket: sequences in the order in which their units are handed out (longest first, so that the
    // launch does not end on a long unit while the other SMs idle); NULL: in index order.
    const int32_t* order;
    // Split calls with a start state: the summary launch copies state_in[unit] here ([unit][64][64] fp32, in
    // the scratch) and every CTA of the main launch takes its start state from the copy, so that nothing
    // reads state_in once the first state_out has been written (state_out may be state_in).  NULL: no copy.
    float* state_copy;
    uint32_t wait_limit_us;                // limit of every device-side wait of the launch (0: the default, 2 s)
    // Checkpoint pass (a summary-variant launch over every segment, used by the gradient): starts from state_in, folds
    // the summaries of the segments before its own (nseg > 1: a plain summary launch has left them in `summaries`) and
    // leaves the state before every chunk, and after the last, in ckpt ([unit][chunks + 1][64][64] bf16, dense
    // sequences) instead of a summary.  The prefill proper fills it too in its CKPT instantiations.  NULL: none.
    // Packed sequences: [H][ckpt_slots][64][64], sequence s of head h from slot
    // cu_seqlens[s] / 64 + 2 s on (its chunks + 1 states fit before the next sequence's first slot), with
    // ckpt_slots = total_T / 64 + 2 S.
    float* ckpt;
    long long ckpt_slots;
    // Balanced persistent launches (PERSIST = 2; dense calls with more units than SMs, state_out given): bal_chunks =
    // chunks per unit.  While at least two units per CTA are left they are handed out whole, unit b + k gridDim to CTA b;
    // the chunks of the rest, in order, are cut into gridDim equal ranges of one to two units each, so a unit may
    // begin in one CTA's range and end in the next one's.  A CTA takes the beginning of such a unit first of all and
    // the end of one last, so the state at the cut is there long before it is wanted: it is handed over in
    // state_out[unit] (which the unit's end overwrites with the final state), announced by four words equal to `nonce`
    // (one per state warp; a number no earlier launch has used) in the first y row after the cut, which that chunk's
    // output overwrites.  The launch is cooperative: every CTA a cut waits for is resident.
    int bal_chunks;
    unsigned long long nonce;
    // Summary launch of a split call: nonzero lets a CTA start late in its segment.  Over a run of tokens in which every
    // channel decays by more than 2^-TRAIL_LOG2 any finite fp32 value, 2^128 at most, falls below half of the smallest
    // subnormal, 2^-150, whatever comes after it: dS forgets what lies before such a run, and D is zero.  So the CTA first
    // sums the decays of its segment's last chunks, TRAIL_CHUNKS at a time and at most TRAIL_LOOKS times, and runs from the
    // last chunk boundary after which every channel has decayed that far, if there is one.  What no finite value survives, a
    // NaN or infinity before that boundary does: see poison_later_segments.
    int trail;
};
constexpr int SUMMARY_FLOATS = 64 + 64 * 64;
constexpr float TRAIL_LOG2 = 280.f;    // (278, and a margin for the rounding of the sums)
constexpr int TRAIL_CHUNKS = 15;       // (two warps each)
constexpr int TRAIL_LOOKS = 6;

// Writes a warp's 16 x 64 fp32 accumulator block (acc[n][0..1] = row g, cols 8n+2q,+1;
// acc[n][2..3] = row g+8) as bf16 into rows row0 .. row0+15 of a 128B-swizzled [rows][64] tile.
__device__ __forceinline__ void store_acc_bf16(uint32_t tile, int row0, const float (&acc)[8][4], int lane)
{
    const int mi = lane >> 3, rr = lane & 7;
    const int row = row0 + rr + 8 * (mi & 1);
#pragma unroll
    for (int m = 0; m < 4; ++m)
        stsm_x4(tile + swz(row, (2 * m + (mi >> 1)) << 4),
                pack_bf16(acc[2 * m][0], acc[2 * m][1]), pack_bf16(acc[2 * m][2], acc[2 * m][3]),
                pack_bf16(acc[2 * m + 1][0], acc[2 * m + 1][1]), pack_bf16(acc[2 * m + 1][2], acc[2 * m + 1][3]));
}
// The same for one half of the columns: acc holds columns 32*HALF .. 32*HALF+31.
template <int HALF>
__device__ __forceinline__ void store_half_bf16(uint32_t tile, int row0, const float (&acc)[4][4], int lane)
{
    const int mi = lane >> 3, rr = lane & 7;
    const int row = row0 + rr + 8 * (mi & 1);
#pragma unroll
    for (int m = 0; m < 2; ++m)
        stsm_x4(tile + swz(row, (2 * (2 * HALF + m) + (mi >> 1)) << 4),
                pack_bf16(acc[2 * m][0], acc[2 * m][1]), pack_bf16(acc[2 * m][2], acc[2 * m][3]),
                pack_bf16(acc[2 * m + 1][0], acc[2 * m + 1][1]), pack_bf16(acc[2 * m + 1][2], acc[2 * m + 1][3]));
}

// acc += the bf16 values of columns 32*HALF .. +31 of a 128B-swizzled [16 rows][64] slab (accumulator layout).
template <int HALF>
__device__ __forceinline__ void add_slab_bf16(float (&acc)[4][4], uint32_t slab, int lane)
{
    const int mi = lane >> 3, rr = lane & 7;
    const int row = rr + 8 * (mi & 1);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        uint32_t w0, w1, w2, w3;     // (rows 0-7, block 2m), (rows 8-15, block 2m), (rows 0-7, block 2m+1), (rows 8-15, block 2m+1)
        ldsm_x4(slab + swz(row, (2 * (2 * HALF + m) + (mi >> 1)) << 4), w0, w1, w2, w3);
        acc[2 * m][0] += bf_lo(w0); acc[2 * m][1] += bf_hi(w0); acc[2 * m][2] += bf_lo(w1); acc[2 * m][3] += bf_hi(w1);
        acc[2 * m + 1][0] += bf_lo(w2); acc[2 * m + 1][1] += bf_hi(w2); acc[2 * m + 1][2] += bf_lo(w3); acc[2 * m + 1][3] += bf_hi(w3);
    }
}

// P' = tril(P, -1) + diag(bonus) on columns 32*HALF .. +31 of one warp's 16 rows (rows 16*SP + g
// and + 8) of the score block.
template <int SP, int HALF>
__device__ __forceinline__ void mask_scores(float (&acc)[4][4], int g, int q, float d_lo, float d_hi)
{
#pragma unroll
    for (int nn = 0; nn < 4; ++nn) {
        const int n = 4 * HALF + nn;
        if (n > 2 * SP + 1) {
            acc[nn][0] = acc[nn][1] = acc[nn][2] = acc[nn][3] = 0.f;         // above the diagonal block
        } else if (n >= 2 * SP) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int il = 8 * (n - 2 * SP) + 2 * q + e;                 // column inside the 16 x 16 diagonal block
                acc[nn][e] = il < g ? acc[nn][e] : (il == g ? d_lo : 0.f);
                acc[nn][2 + e] = il < g + 8 ? acc[nn][2 + e] : (il == g + 8 ? d_hi : 0.f);
            }
        }
    }
}
template <int HALF>
__device__ __forceinline__ void mask_scores_sp(int sp, float (&acc)[4][4], int g, int q, float d_lo, float d_hi)
{
    switch (sp) {
    case 0: mask_scores<0, HALF>(acc, g, q, d_lo, d_hi); break;
    case 1: mask_scores<1, HALF>(acc, g, q, d_lo, d_hi); break;
    case 2: mask_scores<2, HALF>(acc, g, q, d_lo, d_hi); break;
    default: mask_scores<3, HALF>(acc, g, q, d_lo, d_hi); break;
    }
}

// oa, ob += the decay totals of the NQ elementwise warps before this one (slots of 64 floats from `tot`; this lane's
// four channels).  The loads are issued together and the sums formed pairwise, so that the latency is one
// shared-memory round trip plus log2(NQ) additions rather than NQ of each in a row.
template <int NQ>
__device__ __forceinline__ void add_totals(uint32_t tot, float2& oa, float2& ob)
{
    constexpr int NB = NQ < 4 ? NQ : 4;          // at most four slots in flight (registers)
    float2 a[NB], b[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const float4 t4 = ldsf4(tot + 256 * q);
        a[q] = make_float2(t4.x, t4.y); b[q] = make_float2(t4.z, t4.w);
    }
#pragma unroll
    for (int n = NB; n > 1; n = (n + 1) / 2)
#pragma unroll
        for (int q = 0; q < n / 2; ++q) {
            a[q] = add2(a[q], a[n - 1 - q]); b[q] = add2(b[q], b[n - 1 - q]);
        }
    oa = add2(oa, a[0]); ob = add2(ob, b[0]);
    if constexpr (NQ > 4) add_totals<NQ - 4>(tot + 256 * 4, oa, ob);
}

// Token-by-token fp32 recurrence over `valid` tokens of one chunk for one state warp: the warp owns value
// channels 16*sp .. 16*sp+15 for all 64 key channels of the fp32 state copy `scr` ([64][64], row = key
// channel); lane = 16*half + jl works on S[32*half .. +31][16*sp + jl].  Inputs are re-read from global
// memory and y is written there.  The loops are kept rolled: this is the exceptional path, and unrolling
// them costs the fast path registers.
template <bool WITH_OUTPUT>
__device__ __forceinline__ void exact_chunk(float* scr, const Params& p, int h, int sp, int lane, long long first_row,
                                         int valid, size_t C, int col0)
{
    const int half = lane >> 4, j = 16 * sp + (lane & 15);
    float* scol = scr + (32 * half) * 64 + j;
    const float* ug = p.u + h * 64 + 32 * half;
    const bool c2 = p.c2 != 0;
#pragma unroll 1
    for (int t = 0; t < valid; ++t) {
        const size_t ro = (size_t)(first_row + t) * C + col0;
        const float vj = __bfloat162float(p.v[ro + j]);
        float yj = 0.f, cf = 0.f;
#pragma unroll 1
        for (int i = 0; i < 32; i += 2) {
            const uint32_t kw = *reinterpret_cast<const uint32_t*>(p.k + ro + 32 * half + i);
            const uint32_t xw = *reinterpret_cast<const uint32_t*>(p.x + ro + 32 * half + i);
            const float s0 = scol[i * 64], s1 = scol[(i + 1) * 64];
            const float w0 = expf(-expf(bf_lo(xw))), w1 = expf(-expf(bf_hi(xw)));
            float k0 = bf_lo(kw), k1 = bf_hi(kw);
            if (c2) { k0 *= 1.f - w0; k1 *= 1.f - w1; }
            if (WITH_OUTPUT) {
                const uint32_t rw = *reinterpret_cast<const uint32_t*>(p.r + ro + 32 * half + i);
                if (!c2) {
                    cf = fmaf(bf_lo(rw) * ug[i], k0, cf);
                    cf = fmaf(bf_hi(rw) * ug[i + 1], k1, cf);
                }
                yj = fmaf(bf_lo(rw), s0, yj);
                yj = fmaf(bf_hi(rw), s1, yj);
            }
            scol[i * 64] = fmaf(w0, s0, k0 * vj);
            scol[(i + 1) * 64] = fmaf(w1, s1, k1 * vj);
        }
        if (WITH_OUTPUT) {
            yj += __shfl_xor_sync(0xffffffffu, yj, 16);
            cf += __shfl_xor_sync(0xffffffffu, cf, 16);
            if (half == 0) {
                float out = fmaf(cf, vj, yj);
                if (p.u2) out += __bfloat162float(p.u2[ro + j]);
                p.y[ro + j] = __float2bfloat16_rn(out);
            }
        }
    }
}

// Main launch of a split call whose summary launch may have started late in its segments (Params::trail): a segment's state
// that has become non-finite goes on being so, although the summary did not see it.  A CTA whose segment ends like that
// writes NaN over those elements of its summary's dS and says so in the sign of D[1]; every CTA says in the sign of D[0] of
// the summary before its segment that its outputs are written (D is a decay, readers drop the signs).
// Whichever of two CTAs of a unit comes second sees the other's word (a sequentially consistent fence lies between what a CTA
// says and what it reads) and makes the marked columns of the later segment's outputs NaN, and the marked elements of the final
// state and (CKPT) of the segment's checkpoints.  Runs after the CTA's last barrier; without a mark it costs a fence and a load
// of one word per segment, by one warp's lanes at once.  first_slot: the unit's first checkpoint slot.
template <bool CKPT>
__device__ __forceinline__ void poison_later_segments(const Params& p, int unit, int seg, bool marked, int* mark, int* todo, size_t first_slot)
{
    const int tid = threadIdx.x, nseg = p.nseg;
    unsigned* base = reinterpret_cast<unsigned*>(p.summaries) + (size_t)unit * (nseg - 1) * SUMMARY_FLOATS;
    if (tid < 32) {
        // todo: bit g (g < seg): this segment takes the marks of segment g; bit g > seg: segment g takes this one's
        if (tid == 0) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");          // (the outputs and the marked elements before the words)
            if (marked && seg < nseg - 1) atomicOr(base + (size_t)seg * SUMMARY_FLOATS + 1, 0x80000000u);
            if (seg > 0) atomicOr(base + (size_t)(seg - 1) * SUMMARY_FLOATS, 0x80000000u);
        }
        __syncwarp();
        asm volatile("fence.sc.gpu;" ::: "memory");
        unsigned w = 0;
        if (tid < nseg && (tid < seg || (marked && tid > seg)))
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(tid < seg ? base + (size_t)tid * SUMMARY_FLOATS + 1
                                                                                        : base + (size_t)(tid - 1) * SUMMARY_FLOATS) : "memory");
        const unsigned t = __ballot_sync(0xffffffffu, w >> 31);
        if (tid == 0) *todo = (int)t;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    __syncthreads();
    const int t = *todo;
    if (t == 0) return;
    const int seq = unit / p.H, h = unit % p.H;
    const long long row0 = p.cu_seqlens ? p.cu_seqlens[seq] : (long long)seq * p.T;
    const int len = p.cu_seqlens ? p.cu_seqlens[seq + 1] - p.cu_seqlens[seq] : p.T;
    const float nan = __int_as_float(0x7fc00000);
    for (int g = 0; g < nseg; ++g) {
        if (!(t >> g & 1)) continue;
        const int from = g < seg ? g : seg, to = g < seg ? seg : g;
        const float* ds = reinterpret_cast<const float*>(base + (size_t)from * SUMMARY_FLOATS + 64);
        const int first = min(len, to * p.seg_chunks * L), end = to == nseg - 1 ? len : min(len, first + p.seg_chunks * L);
        // the states before the segment's chunks, and after the last one of the unit
        const int ck_first = (first + L - 1) / L, ck_end = (end + L - 1) / L + (to == nseg - 1 ? 1 : 0);
        __syncthreads();
        if (tid < 64) mark[tid] = 0;
        __syncthreads();
        for (int i = tid; i < 4096; i += blockDim.x) {
            const float v = __ldcg(ds + i);
            if (v != v) {
                mark[i & 63] = 1;
                if (to == nseg - 1 && p.state_out) p.state_out[(size_t)unit * 4096 + i] = nan;
                if (CKPT)
                    for (int c = ck_first; c < ck_end; ++c)
                        reinterpret_cast<__nv_bfloat16*>(p.ckpt)[(first_slot + c) * 4096 + i] = __float2bfloat16_rn(nan);
            }
        }
        __syncthreads();
        for (long long i = (long long)first * 64 + tid; i < (long long)end * 64; i += blockDim.x)
            if (mark[i & 63]) p.y[(size_t)(row0 + (i >> 6)) * p.H * 64 + h * 64 + (i & 63)] = __float2bfloat16_rn(nan);
    }
}

// ---------------------------------------------------------------- the kernel
// SUMMARY = false: the prefill proper.  SUMMARY = true: the first pass of a split call, which only
// carries the state over a segment from a zero start (no r, no scores, no outputs: the score warps and
// the second MMA warp idle, the output warps only serve the token-by-token path) and writes the
// segment's summary.
// C2 = true: the Finch-C2 form (keys times one minus their decay, no bonus, optional second-value vector).
// PERSIST != 0: the CTA walks a stream of units (see Params::n_units); the producer warp leaves a descriptor per
// chunk and two end markers, which every role passes down its own signalling path before it leaves.  PERSIST = 2: the
// stream may begin and end inside a unit (see Params::bal_chunks).
// CKPT = true (launches of the prefill proper): the state before every chunk and after the last one is also left in
// Params::ckpt, for the gradient call that follows a training step's forward pass.
// TRAIL = true (main launches of split calls): the summary launch may have started late in its segments (see Params::trail).
template <bool SUMMARY, bool C2, int PERSIST = 0, bool CKPT = false, bool TRAIL = false>
__global__ void __launch_bounds__(THREADS, 1)
wkv6_chunked_kernel(const __grid_constant__ CUtensorMap tm_r, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_x,
                    const __grid_constant__ CUtensorMap tm_y16, const __grid_constant__ CUtensorMap tm_u2_16,
                    const Params p, const __grid_constant__ CUtensorMap tm_ck16)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const uint32_t abort_flag = sbase + OFF_ABORT;           // shared addresses of the abort word and the safety flags
    auto safe_at = [&](int sd) { return lds32(sbase + OFF_SAFE + 4 * sd) != 0; };
    auto bar = [&](int i) { return sbase + OFF_BAR + 8 * i; };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // first pass of a split call: the second launch (enqueued with programmatic stream serialisation) may set up and
    // fill its rings while this one runs; its state warps wait for this grid's results before they read them.
    // Unsplit prefills (EARLY) start early too, behind whatever kernel is ahead of them, and wait as a whole once they are set
    // up: 1.2 us of every call (320 tokens in 80 units 6.4 -> 5.1 us, 333 tokens 11.2 -> 10.0, LayerNorm behind 278 tokens 11.4 -> 9.7).
    // Not the balanced and the checkpointing variants, whose code comes out 1-2 % slower with the two instructions
    // (Finch-C2, 5 x 2011 tokens: 78.4 -> 79.9; packed training pair 615 -> 618).
    constexpr bool EARLY = !SUMMARY && PERSIST != 2 && !CKPT;
    if (SUMMARY || EARLY) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int gsegs = (SUMMARY && !p.ckpt) ? p.nseg - 1 : p.nseg;      // segments per unit that this launch covers
    const int unit = blockIdx.x / gsegs, seg = blockIdx.x % gsegs;
    const int seq = unit / p.H, h = unit % p.H;
    long long row0;
    int len;
    if (p.cu_seqlens) {
        if (EARLY && !PERSIST && p.nseg == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
        row0 = p.cu_seqlens[seq];
        len = p.cu_seqlens[seq + 1] - p.cu_seqlens[seq];
    } else {
        row0 = (long long)seq * p.T;
        len = p.T;
    }
    if (p.nseg > 1) {                                      // this CTA's segment of the sequence
        const int first = min(len, seg * p.seg_chunks * L);
        row0 += first;
        len = (seg == p.nseg - 1) ? len - first : min(len - first, p.seg_chunks * L);
    }
    int trail_cut = 0;                     // (see Params::trail) chunks of the segment that need not be run
    if constexpr (SUMMARY) {
        // only whole, full segments (of which all but the last chunks may go); two warps per chunk sum it, 32 tokens each, with
        // all their loads in flight: lane = 4 channels (lane % 16) of every other row
        const int n_full = len / L;
        if (p.trail && len % L == 0 && n_full > 1) {
            float* tot = reinterpret_cast<float*>(smem);           // [TRAIL_CHUNKS][2][64] (the ring: nothing has been loaded yet)
            float a0 = 0.f, a1 = 0.f;                              // every warp finds the same answer: two channels per lane
            for (int k0 = 0; k0 < min(TRAIL_LOOKS * TRAIL_CHUNKS, n_full - 1) && !trail_cut; k0 += TRAIL_CHUNKS) {
                const int look = min(TRAIL_CHUNKS, n_full - 1 - k0), cw = n_full - 1 - k0 - (warp >> 1);      // (this warp's chunk)
                if (warp < 2 * look) {
                    const __nv_bfloat16* xp = p.x + (size_t)(row0 + (long long)cw * L + 32 * (warp & 1) + (lane >> 4)) * ((size_t)p.H * 64) + h * 64 + 4 * (lane & 15);
                    uint2 w[L / 4];
#pragma unroll
                    for (int t = 0; t < L / 4; ++t) w[t] = *reinterpret_cast<const uint2*>(xp + (size_t)(2 * t) * ((size_t)p.H * 64));
                    float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int t = 0; t < L / 4; ++t) {
                        e[0] += ex2(fmaf(bf_lo(w[t].x), LOG2E, LOG2_LOG2E)); e[1] += ex2(fmaf(bf_hi(w[t].x), LOG2E, LOG2_LOG2E));
                        e[2] += ex2(fmaf(bf_lo(w[t].y), LOG2E, LOG2_LOG2E)); e[3] += ex2(fmaf(bf_hi(w[t].y), LOG2E, LOG2_LOG2E));
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] += __shfl_xor_sync(0xffffffffu, e[i], 16);
                    if (lane < 16) *reinterpret_cast<float4*>(tot + warp * 64 + 4 * lane) = make_float4(e[0], e[1], e[2], e[3]);
                }
                __syncthreads();
                for (int k = 0; k < look; ++k) {                   // chunks from the last one back
                    a0 += tot[k * 128 + 2 * lane] + tot[k * 128 + 64 + 2 * lane]; a1 += tot[k * 128 + 2 * lane + 1] + tot[k * 128 + 64 + 2 * lane + 1];
                    if (__all_sync(0xffffffffu, a0 > TRAIL_LOG2 && a1 > TRAIL_LOG2)) { trail_cut = n_full - 1 - k0 - k; break; }     // (false for NaN)
                }
                __syncthreads();                                   // (the sums are read before they, or the ring, are written again)
                // (decays that have not come their share of the way are too slow for the looks that are left)
                const float share = TRAIL_LOG2 / TRAIL_LOOKS * (float)(k0 / TRAIL_CHUNKS + 1);
                if (!__all_sync(0xffffffffu, a0 > 0.9f * share && a1 > 0.9f * share)) break;
            }
            row0 += (long long)trail_cut * L;
            len -= trail_cut * L;
            fence_proxy_async();
        }
    }
    const int nchunks = PERSIST ? 0 : (len + L - 1) / L;
    // checkpoint slots of this unit: the first one, and how many chunks the whole sequence has
    auto ckpt_slot = [&](int c_abs) -> size_t {       // (the packed form recomputes what it needs: nothing stays live for it)
        if (p.cu_seqlens) {
            const int sq = unit / p.H, hh = unit - sq * p.H;
            return (size_t)hh * p.ckpt_slots + (size_t)(p.cu_seqlens[sq] >> 6) + 2 * (size_t)sq + c_abs;
        }
        return (size_t)unit * ((p.T + L - 1) / L + 1) + c_abs;
    };
    auto ckpt_chunks = [&]() -> int {                 // chunks of the whole sequence (this CTA may hold one segment of it)
        if (p.cu_seqlens) {
            const int sq = unit / p.H;
            return (p.cu_seqlens[sq + 1] - p.cu_seqlens[sq] + L - 1) / L;
        }
        return (p.T + L - 1) / L;
    };
    const int col0 = h * 64;
    const size_t C = (size_t)p.H * 64;
    static_assert(!(PERSIST && SUMMARY), "the summary pass is a single-unit launch");
    static_assert(!(CKPT && SUMMARY), "the summary pass keeps its checkpoints by Params::ckpt");
    static_assert(!(TRAIL && (PERSIST || SUMMARY)), "the main launch of a split call");
    constexpr bool BAL = PERSIST == 2;
    constexpr bool PAIR = C2 && !SUMMARY && (BAL || (CKPT && !PERSIST));          // two second-value slabs per output warp (see there)

    // One chunk of this CTA's work.  Single-unit launches derive it from the chunk index; persistent launches
    // read the descriptor the producer warp left for the chunk, which is visible to any warp that has waited
    // on a barrier downstream of the chunk's "full" barrier.
    struct Chunk { int row; int valid; int unit; int h; int rem; bool first; bool last; bool end; };
    auto chunk_at = [&](int c) -> Chunk {
        Chunk ck;
        if constexpr (PERSIST) {
            int4 d;
            asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w) : "r"(sbase + OFF_DESC + 16 * (c & (NSIDE - 1))) : "memory");
            ck.row = d.x; ck.valid = d.y & 0xff; ck.unit = d.z; ck.rem = d.w;
            ck.h = BAL ? d.y >> 16 : (int)((unsigned)d.y >> 16);      // (a balanced call has fewer than five units per SM: no sign; spills)
            ck.first = (d.y & DESC_FIRST) != 0; ck.last = BAL ? (d.y & DESC_LAST) != 0 : d.w == 0; ck.end = (d.y & DESC_END) != 0;
        } else {
            ck.row = (int)(row0 + (long long)c * L); ck.valid = min(L, len - c * L); ck.unit = unit; ck.h = h;
            ck.rem = nchunks - 1 - c; ck.first = c == 0; ck.last = ck.rem == 0; ck.end = false;
        }
        return ck;
    };
    auto chunk_continues = [&](int c) -> bool {      // (balanced launches) a piece of a unit that another CTA began
        return (lds32(sbase + OFF_DESC + 16 * (c & (NSIDE - 1)) + 4) & DESC_CONT) != 0;
    };
    auto chunk_is_end = [&](int c) -> bool {
        if constexpr (PERSIST) return (lds32(sbase + OFF_DESC + 16 * (c & (NSIDE - 1)) + 4) & DESC_END) != 0;
        return false;
    };

    if (tid == 0) {
        for (int i = 0; i < N_ESET * NS; ++i) mbar_init(bar(BAR_FULL_RKV + i), 1);
        for (int i = 0; i < STAGE_STEP; ++i) mbar_arrive(bar(BAR_FULL_RKV + NS + i));      // (see STAGE_STEP)
        for (int i = 0; i < NS; ++i) {
            mbar_init(bar(BAR_EMPTY_RKV + i), 1);                  // the commit after the last product that reads the stage
            mbar_init(bar(BAR_RK_READY + i), N_EW);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(BAR_S_READY + i), N_GW);
            mbar_init(bar(BAR_PP_READY + i), N_GW);
            mbar_init(bar(BAR_F_FULL + i), 1);
            mbar_init(bar(BAR_F_EMPTY + i), 2 * N_GW);              // state + score warps (summary pass: state + output warps)
            mbar_init(bar(BAR_B_DONE + i), 1);
            mbar_init(bar(BAR_Y_EMPTY + i), N_GW);
        }
        for (int i = 0; i < N_ESET; ++i) mbar_init(bar(BAR_ESYNC + i), N_EW);
        mbar_init(bar(BAR_SSYNC), N_GW);
        mbar_init(bar(BAR_SPRE), N_GW);
        mbar_init(bar(BAR_FB_READY), N_GW);
        mbar_init(bar(BAR_FB_DONE), N_GW);
        for (int i = 0; i < (PAIR ? 2 : 1) * N_GW; ++i) mbar_init(bar(BAR_U2 + i), 1);
        if (C2 && BAL)
            for (int i = 0; i < NSIDE; ++i) sts32(sbase + OFF_DESC + 16 * i + 4, DESC_TAG);        // (of the turn before the first)
        sts32(abort_flag, 0u);
        sts32(abort_flag + 4, p.wait_limit_us ? p.wait_limit_us : WAIT_LIMIT_US);
        if (TRAIL) sts32(sbase + OFF_MARK, 0u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == WARP_MMA_F) tmem_alloc(sbase + OFF_TMEM, TM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = lds32(sbase + OFF_TMEM);
    if (EARLY && (PERSIST || p.nseg == 1)) asm volatile("griddepcontrol.wait;" ::: "memory");

    // (producer lane) leaves the descriptor of chunk gc of the stream.  Roles that wait on a barrier downstream of the
    // chunk's copies find it complete; the tag, written last, is for the one that looks at it earlier (desc_wait).
    auto put_desc = [&](int gc, int row, int meta, int u, int rem) {
        const uint32_t d = sbase + OFF_DESC + 16 * (gc & (NSIDE - 1));
        const int tag = ((gc / NSIDE) & 1) * DESC_TAG;
        if (C2 && BAL) meta |= tag ^ DESC_TAG;
        asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(d), "r"(row), "r"(meta), "r"(u), "r"(rem) : "memory");
        if (C2 && BAL) asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(d + 4), "r"(meta ^ DESC_TAG) : "memory");
    };

    if (warp == 0) {
        // ============================== TMA producer ==============================
        auto full_bar = [&](int c) { return bar(BAR_FULL_RKV + (c & 1) * NS + STAGE_STEP * c % NS); };
        auto full_parity = [&](int c) { return (uint32_t)(((c >> 1) + (c & 1) * STAGE_STEP) / NS & 1); };
        if constexpr (PERSIST) {
            int gc = 0, real_end = -1;               // chunks of the stream issued so far; index of the first end marker
            int s = 0, ph = 1;                       // ring stage and the parity of its previous release
            bool alive = true;
            for (int k = 0; alive; ++k) {
                int u = 0, c0 = 0, c1 = 0;               // the next piece: chunks c0 .. c1-1 of unit u (balanced launches)
                if constexpr (BAL) {
                    // First the beginning of the unit this CTA's range ends in, then whole units, last the end of the unit
                    // the range begins in.  (32-bit products: the host balances only calls whose chunk counts allow it.)
                    const unsigned G = gridDim.x, nc = p.bal_chunks, rounds = p.n_units / G - 1, R = p.n_units - rounds * G, bi = blockIdx.x;
                    const unsigned b0 = R * nc * bi / G, b1 = R * nc * (bi + 1) / G;
                    const unsigned head = b1 % nc, tail = b0 % nc;
                    int kk = k - (head != 0);
                    c1 = nc;
                    // Which unit: neighbouring heads share lines of memory, so units processed at the same time get
                    // neighbouring indices.  The cut ones come first, by CTA (their beginnings all start the launch and
                    // their ends all close it), then the whole ones by the time at which their CTA starts them.
                    auto cuts_before = [&](unsigned n) {                                     // cuts at the ends of the first n CTAs
                        int cuts = 0;
                        for (unsigned b = lane; b < n; b += 32) cuts += R * nc * (b + 1) / G % nc != 0;
                        return (unsigned)__reduce_add_sync(0xffffffffu, cuts);
                    };
                    if (kk < 0) { u = rounds * G + cuts_before(bi); c1 = head; }
                    else if (kk < (int)rounds) u = bi + kk * G;
                    else {
                        kk -= rounds;
                        const bool whole = b1 / nc > (b0 + nc - 1) / nc;                     // (a range holds at most one whole unit)
                        if (whole && kk == 0) {
                            int before = 0;
                            for (unsigned b = lane; b < G; b += 32) {
                                const unsigned e0 = R * nc * b / G, e1 = R * nc * (b + 1) / G, eh = e1 % nc;
                                before += e1 / nc > (e0 + nc - 1) / nc && (eh < head || (eh == head && b < bi));
                            }
                            u = rounds * G + cuts_before(G) + __reduce_add_sync(0xffffffffu, before);
                        } else if (kk == (whole ? 1 : 0) && tail != 0) {
                            u = rounds * G + cuts_before(bi) - 1; c0 = tail;
                        } else break;
                    }
                } else if (p.ticket) {
                    if (lane == 0) u = (int)atomicAdd(p.ticket, 1u);
                    u = __shfl_sync(0xffffffffu, u, 0);
                } else {
                    u = blockIdx.x + k * gridDim.x;
                }
                if (u >= p.n_units) break;
                int useq = u / p.H;
                const int uh = u % p.H;
                if (p.ticket && p.order) {               // the ticket counts through the sequences longest first
                    useq = p.order[useq];
                    u = useq * p.H + uh;
                }
                long long urow0;
                int ulen;
                if (p.cu_seqlens) {
                    urow0 = p.cu_seqlens[useq];
                    ulen = p.cu_seqlens[useq + 1] - p.cu_seqlens[useq];
                } else {
                    urow0 = (long long)useq * p.T;
                    ulen = p.T;
                }
                const int unch = (ulen + L - 1) / L;
                if (unch == 0) {
                    // empty sequence: its state passes through; no chunk enters the stream
                    if (p.state_out && p.state_out != p.state_in)
                        for (int i = lane; i < 4096; i += 32)
                            p.state_out[(size_t)u * 4096 + i] = p.state_in ? p.state_in[(size_t)u * 4096 + i] : 0.f;
                    if constexpr (CKPT) {                    // (its only checkpoint, in the packed layout of ckpt_slot above)
                        const size_t slot = (size_t)uh * p.ckpt_slots + (size_t)(p.cu_seqlens[useq] >> 6) + 2 * (size_t)useq;
                        for (int i = lane; i < 4096; i += 32)
                            reinterpret_cast<__nv_bfloat16*>(p.ckpt)[slot * 4096 + i] = __float2bfloat16_rn(p.state_in ? p.state_in[(size_t)u * 4096 + i] : 0.f);
                    }
                    continue;
                }
                if (!BAL) c1 = unch;
                if (p.state_in && (!BAL || c0 == 0)) {
                    // the state warps read this unit's start state a few chunks from now: have it in L2 by then
                    const char* sp0 = reinterpret_cast<const char*>(p.state_in + (size_t)u * 4096);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(sp0 + 128 * (lane + 32 * i)));
                }
                for (int c = c0; c < c1; ++c, ++gc) {
                    if (gc >= NS && !mbar_wait_warp(bar(BAR_EMPTY_RKV + s), ph, abort_flag)) { alive = false; break; }
                    const int row = (int)(urow0 + (long long)c * L);
                    const uint32_t dst = sbase + OFF_RING + s * STAGE;
                    if (elect_one()) {
                        int meta = min(L, ulen - c * L) | (c == c0 ? DESC_FIRST : 0) | (int)((unsigned)uh << 16);
                        if (BAL) meta |= (c == c0 && c0 > 0 ? DESC_CONT : 0) | (c == c1 - 1 ? DESC_LAST : 0);
                        put_desc(gc, row, meta, u, unch - 1 - c);
                        const uint32_t full = bar(BAR_FULL_RKV + (gc & 1) * NS + s);
                        mbar_expect_tx(full, STAGE);                       // (release: the descriptor is visible to the waiters)
                        tma_load_2d(dst, &tm_x, uh * 64, row, full);
                        tma_load_2d(dst + TILE, &tm_r, uh * 64, row, full);
                        tma_load_2d(dst + 2 * TILE, &tm_k, uh * 64, row, full);
                        tma_load_2d(dst + 3 * TILE, &tm_v, uh * 64, row, full);
                    }
                    __syncwarp();
                    next_stage(s, ph);
                }
            }
            if (alive) {
                // two end markers, one for each elementwise set; each role hands them on and leaves
                real_end = gc;
                for (int e = 0; e < 2 && alive; ++e, ++gc) {
                    if (gc >= NS && !mbar_wait_warp(bar(BAR_EMPTY_RKV + s), ph, abort_flag)) { alive = false; break; }
                    if (elect_one()) {
                        put_desc(gc, 0, DESC_END, 0, 0);
                        mbar_arrive(bar(BAR_FULL_RKV + (gc & 1) * NS + s)); // no copy: the arrival alone completes the phase
                    }
                    __syncwarp();
                    next_stage(s, ph);
                }
            }
            // Do not leave while copies into this CTA's shared memory may still be in flight.  A stage that an end
            // marker re-used was released by its consumers first, so only the chunks after those need the wait.
            const int issued = real_end >= 0 ? real_end : gc;
            const int from = (real_end >= 0 && alive) ? max(0, issued - NS + 2) : max(0, issued - NS);
            for (int c = from; c < issued; ++c)
                mbar_wait_warp(full_bar(c), full_parity(c), abort_flag, false);
        } else {
            int issued = 0;
            int s = 0, ph = 1;                       // ring stage and the parity of its previous release
            int row = (int)row0;
            for (int c = 0; c < nchunks; ++c, row += L) {
                if (c >= NS && !mbar_wait_warp(bar(BAR_EMPTY_RKV + s), ph, abort_flag)) break;
                const uint32_t dst = sbase + OFF_RING + s * STAGE;
                if (elect_one()) {
                    const uint32_t full = bar(BAR_FULL_RKV + (c & 1) * NS + s);
                    mbar_expect_tx(full, SUMMARY ? 3 * TILE : STAGE);
                    tma_load_2d(dst, &tm_x, col0, row, full);
                    if (!SUMMARY) tma_load_2d(dst + TILE, &tm_r, col0, row, full);
                    tma_load_2d(dst + 2 * TILE, &tm_k, col0, row, full);
                    tma_load_2d(dst + 3 * TILE, &tm_v, col0, row, full);
                }
                __syncwarp();
                issued = c + 1;
                next_stage(s, ph);
            }
            // do not leave while copies into this CTA's shared memory may still be in flight
            for (int c = max(0, issued - NS); c < issued; ++c)
                mbar_wait_warp(full_bar(c), full_parity(c), abort_flag, false);
        }
    } else if (warp == WARP_MMA_F) {
        // ============================== MMA issuer, input-only products ==============================
        // P_c = R^ K^^T (M = t, N = i, K = c: both operands K-major) and dS_c = K^^T V (M = c, N = j,
        // K = i: both MN-major), interleaved: consecutive tcgen05.mma on one accumulator wait for each
        // other, different accumulators pipeline.
        int s = 0, ph = 0;                       // ring stage and its phase bit
        for (int c = 0; PERSIST || c < nchunks; ++c) {
            const int tb = c & 1, pt = (c >> 1) & 1;
            if (!mbar_wait_warp(bar(BAR_RK_READY + s), ph, abort_flag)) break;
            if (c >= 2 && !mbar_wait_warp(bar(BAR_F_EMPTY + tb), pt ^ 1, abort_flag)) break;
            if (PERSIST && chunk_is_end(c)) {        // hand the end marker to the state and score warps
                if (elect_one()) mbar_arrive(bar(BAR_F_FULL + tb));
                __syncwarp();
                break;
            }
            const bool safe = safe_at(c & (NSIDE - 1));
            const uint32_t tr = sbase + OFF_RING + s * STAGE + TILE;
            tc_fence_after();
            if (elect_one()) {
                if (safe) {
                    const uint64_t dr = smem_desc(tr), dk = smem_desc(tr + TILE), dv = smem_desc(tr + 2 * TILE);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        if (!SUMMARY)
                            tc_mma(tmem + TM_P + 64 * tb, dr + (uint64_t)(2 * kk), dk + (uint64_t)(2 * kk), IDESC_K_K, kk > 0);
                        tc_mma(tmem + TM_DS + 64 * tb, dk + (uint64_t)(128 * kk), dv + (uint64_t)(128 * kk), IDESC_MN_MN, kk > 0);
                    }
                }
                tc_commit(bar(BAR_F_FULL + tb));
                if (SUMMARY) tc_commit(bar(BAR_EMPTY_RKV + s));    // no other product reads the stage
            }
            __syncwarp();
            next_stage(s, ph);
        }
    } else if (warp == WARP_MMA_B) {
        // ============================== MMA issuer, state-dependent products ==============================
        // Y0_c = R^ S_0 (M = t, N = j, K = c) and PV_c = P' V (M = t, N = j, K = i): A K-major, B MN-major.
        // The masked scores of chunk c exist only after P_c completed, so every product that reads
        // ring stage s is complete when these complete: the last commit releases the stage.
        int s = 0;
        for (int c = 0; PERSIST || c < (SUMMARY ? 0 : nchunks); ++c) {
            const int tb = c & 1, pt = (c >> 1) & 1;
            if (c >= 2 && !mbar_wait_warp(bar(BAR_Y_EMPTY + tb), pt ^ 1, abort_flag)) break;
            if (!mbar_wait_warp(bar(BAR_S_READY + tb), pt, abort_flag)) break;
            if (!mbar_wait_warp(bar(BAR_PP_READY + tb), pt, abort_flag)) break;
            if (PERSIST && chunk_is_end(c)) {        // hand the end marker to the output warps
                if (elect_one()) mbar_arrive(bar(BAR_B_DONE + tb));
                __syncwarp();
                break;
            }
            const bool safe = safe_at(c & (NSIDE - 1));
            const uint32_t tr = sbase + OFF_RING + s * STAGE + TILE;
            tc_fence_after();
            if (elect_one()) {
                if (safe) {
                    const uint64_t dr = smem_desc(tr), dv = smem_desc(tr + 2 * TILE);
                    const uint64_t ds = smem_desc(sbase + OFF_SB + tb * TILE), dp = smem_desc(sbase + OFF_PP + tb * TILE);
#pragma unroll
                    // one accumulator: Y = [R^ | P'] [S_0 ; V], the state part first (its operands are ready earlier)
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma(tmem + TM_Y + 64 * tb, dr + (uint64_t)(2 * kk), ds + (uint64_t)(128 * kk), IDESC_K_MN, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma(tmem + TM_Y + 64 * tb, dp + (uint64_t)(2 * kk), dv + (uint64_t)(128 * kk), IDESC_K_MN, 1);
                }
                tc_commit(bar(BAR_B_DONE + tb));
                tc_commit(bar(BAR_EMPTY_RKV + s));
            }
            __syncwarp();
            s += STAGE_STEP;
            if (s >= NS) s -= NS;
        }
    } else if (warp < WARP_P0) {
        // ============================== state warps ==============================
        const int sp = warp & 3;                 // tensor-memory sub-partition: key channels 16*sp .. 16*sp+15
        const int g = lane >> 2, q = lane & 3;
        const int c_lo = 16 * sp + g;
        const size_t sb = (size_t)unit * 4096;
        // S[c][j] in accumulator layout: st[n][0..1] = (c_lo, j = 8n+2q, +1), st[n][2..3] = (c_lo+8, same j)
        float st[8][4];
        // the start states of this launch: the caller's, or (main launch of a split call) the summary launch's copy
        const float* s_src = (!SUMMARY && p.state_copy) ? p.state_copy : p.state_in;
        auto load_state = [&](size_t base) {         // this lane's part of the start state of a unit (zero without one)
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                if ((!SUMMARY || p.ckpt) && s_src) {
                    const float2 lo = *reinterpret_cast<const float2*>(s_src + base + (size_t)c_lo * 64 + 8 * n + 2 * q);
                    const float2 hi = *reinterpret_cast<const float2*>(s_src + base + (size_t)(c_lo + 8) * 64 + 8 * n + 2 * q);
                    st[n][0] = lo.x; st[n][1] = lo.y; st[n][2] = hi.x; st[n][3] = hi.y;
                } else {
                    st[n][0] = st[n][1] = st[n][2] = st[n][3] = 0.f;
                }
            }
        };
        if (SUMMARY && seg == 0 && p.state_in && p.state_copy) {
            // first pass of a split call: keep the unit's start state for the second pass (see Params::state_copy)
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                const size_t lo = sb + (size_t)c_lo * 64 + 8 * n + 2 * q, hi = sb + (size_t)(c_lo + 8) * 64 + 8 * n + 2 * q;
                *reinterpret_cast<float2*>(p.state_copy + lo) = *reinterpret_cast<const float2*>(p.state_in + lo);
                *reinterpret_cast<float2*>(p.state_copy + hi) = *reinterpret_cast<const float2*>(p.state_in + hi);
            }
        }
        auto store_to = [&](float* dst) {            // this lane's part of the state into a [64][64] fp32 block
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                *reinterpret_cast<float2*>(dst + (size_t)c_lo * 64 + 8 * n + 2 * q) = make_float2(st[n][0], st[n][1]);
                *reinterpret_cast<float2*>(dst + (size_t)(c_lo + 8) * 64 + 8 * n + 2 * q) = make_float2(st[n][2], st[n][3]);
            }
        };
        auto store_state = [&](size_t base) { store_to(p.state_out + base); };
        // a checkpoint: the state rounded to bf16, [64][64] row-major (8 KB: as the gradient's tensor-core operand reads it)
        auto store_ckpt = [&](size_t slot) {
            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.ckpt) + slot * 4096;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                *reinterpret_cast<uint32_t*>(dst + (size_t)c_lo * 64 + 8 * n + 2 * q) = pack_bf16(st[n][0], st[n][1]);
                *reinterpret_cast<uint32_t*>(dst + (size_t)(c_lo + 8) * 64 + 8 * n + 2 * q) = pack_bf16(st[n][2], st[n][3]);
            }
        };
        // second launch of a split call: the summaries and the start-state copy are the first launch's
        if (!SUMMARY && !PERSIST && p.nseg > 1) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!PERSIST) load_state(sb);
        if (!SUMMARY || p.ckpt) {
            // start state of a later segment: fold the summaries of the segments before it, in order
            for (int gg = 0; gg < seg; ++gg) {
                const float* sm = p.summaries + ((size_t)unit * (p.nseg - 1) + gg) * SUMMARY_FLOATS;
                float d_lo = sm[c_lo], d_hi = sm[c_lo + 8];
                if (TRAIL) { d_lo = fabsf(d_lo); d_hi = fabsf(d_hi); }               // (signs: see poison_later_segments)
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    const float2 lo = *reinterpret_cast<const float2*>(sm + 64 + c_lo * 64 + 8 * n + 2 * q);
                    const float2 hi = *reinterpret_cast<const float2*>(sm + 64 + (c_lo + 8) * 64 + 8 * n + 2 * q);
                    st[n][0] = fmaf(d_lo, st[n][0], lo.x); st[n][1] = fmaf(d_lo, st[n][1], lo.y);
                    st[n][2] = fmaf(d_hi, st[n][2], hi.x); st[n][3] = fmaf(d_hi, st[n][3], hi.y);
                }
            }
        }
        float dprod_lo = 1.f, dprod_hi = 1.f;    // summary pass: decay product of the segment for this lane's two rows
        int fb_uses = 0;                         // chunks that took the token-by-token path so far
        // Checkpoints of the chunk-start states: the bf16 copy of the state in its operand tile (the pair of tiles is
        // idle in a summary pass and written for the checkpoints' sake there) is what the gradient reads, so each state
        // warp sends its 16 rows of the tile to the checkpoint array by TMA (tm_ck16: the array as [slots * 64][64]).
        constexpr bool CK_TMA = CKPT || SUMMARY;
        const bool ck_on = CKPT || (SUMMARY && p.ckpt);
        auto ckpt_tile = [&](int tile, size_t slot) {    // after the tile's rows are written, fenced and the warp synchronised
            if (lane == 0) {
                tma_store_2d(&tm_ck16, 0, (int)(slot * 64) + 16 * sp, sbase + OFF_SB + tile * TILE + 16 * sp * 128);
                bulk_commit();
            }
        };
        if (!PERSIST && !SUMMARY && nchunks > 0) {
            store_acc_bf16(sbase + OFF_SB, 16 * sp, st, lane);
            fence_proxy_async();
            __syncwarp();
            mbar_arrive_if(bar(BAR_S_READY), lane == 0);
            if (CKPT) ckpt_tile(0, ckpt_slot(seg * p.seg_chunks));
        }
        if (SUMMARY && ck_on && nchunks > 0) {
            store_acc_bf16(sbase + OFF_SB, 16 * sp, st, lane);
            fence_proxy_async();
            __syncwarp();
            ckpt_tile(0, ckpt_slot(seg * p.seg_chunks));
        }
        int pslot = 0;                           // (persistent launches) checkpoint slot of the current chunk's start state
        for (int c = 0; PERSIST || c < nchunks; ++c) {
            const int tb = c & 1, pt = (c >> 1) & 1, sd = c & (NSIDE - 1);
            if (!mbar_wait(bar(BAR_F_FULL + tb), pt, abort_flag)) break;
            tc_fence_after();
            const Chunk ck = chunk_at(c);
            if (PERSIST && ck.end) {
                // Hand the end marker to the issuer of the state-dependent products, under the same condition as a
                // real operand tile (the products of chunk c-2 are done): the issuer has then consumed this barrier's
                // previous phase, so the marker's arrival cannot run two phases ahead of its wait.
                if (c >= 2 && !mbar_wait(bar(BAR_B_DONE + tb), ((c - 2) >> 1) & 1, abort_flag)) break;
                __syncwarp();
                mbar_arrive_if(bar(BAR_S_READY + tb), lane == 0);
                break;
            }
            if (PERSIST && ck.first) {
                // a new unit starts with this chunk: its state replaces the registers, and the operand tile of
                // this chunk (last read by the products of chunk c-2) takes its bf16 copy
                if (BAL && chunk_continues(c)) {
                    // ... or continues one whose beginning another CTA has: the state at the cut, from state_out
                    bool ok = true;
                    if (lane == 0) {
                        ok = word_wait(reinterpret_cast<const unsigned long long*>(p.y + (size_t)ck.row * C + ck.h * 64) + sp, p.nonce, abort_flag);
                        asm volatile("fence.proxy.async.global;" ::: "memory");       // (the y tile that replaces the word goes by TMA)
                    }
                    if (!__all_sync(0xffffffffu, ok)) break;
                    const float* src = p.state_out + (size_t)ck.unit * 4096 + 2 * q;
#pragma unroll
                    for (int n = 0; n < 8; ++n) {
                        const float2 lo = __ldcg(reinterpret_cast<const float2*>(src + (size_t)c_lo * 64 + 8 * n));
                        const float2 hi = __ldcg(reinterpret_cast<const float2*>(src + (size_t)(c_lo + 8) * 64 + 8 * n));
                        st[n][0] = lo.x; st[n][1] = lo.y; st[n][2] = hi.x; st[n][3] = hi.y;
                    }
                } else {
                    load_state((size_t)ck.unit * 4096);
                }
                if (c >= 2 && !mbar_wait(bar(BAR_B_DONE + tb), ((c - 2) >> 1) & 1, abort_flag)) break;
                if (CKPT) {
                    const int useq = ck.unit / p.H;
                    if (p.cu_seqlens) pslot = (int)((ck.unit - useq * p.H) * p.ckpt_slots) + (p.cu_seqlens[useq] >> 6) + 2 * useq;
                    else pslot = ck.unit * ((p.T + L - 1) / L + 1) + (BAL ? p.bal_chunks - 1 - ck.rem : 0);
                    if (lane == 0) bulk_wait_read<1>();      // the checkpoint copy of chunk c - 2 has finished reading this tile
                    __syncwarp();
                }
                store_acc_bf16(sbase + OFF_SB + tb * TILE, 16 * sp, st, lane);
                fence_proxy_async();
                __syncwarp();
                mbar_arrive_if(bar(BAR_S_READY + tb), lane == 0);
                if (CKPT) ckpt_tile(tb, pslot);
            }
            bool next_tile_free = c == 0;        // the products of chunk c-1 have finished reading operand tile tb^1
            const uint32_t dl = sbase + OFF_DL + 4 * (sd * 64 + c_lo);
            const float d_lo = ldsf(dl), d_hi = ldsf(dl + 32);        // 2^{a_L} of this lane's two rows
            if (SUMMARY) { dprod_lo *= d_lo; dprod_hi *= d_hi; }
            if (safe_at(sd)) {
                // ---- S <- diag(2^{a_L}) (S + K^^T V)
                const float2 dlo2 = make_float2(d_lo, d_lo), dhi2 = make_float2(d_hi, d_hi);
                const uint32_t ta = tmem + ((uint32_t)(32 * sp) << 16) + TM_DS + 64 * tb;
#pragma unroll
                for (int qt = 0; qt < 4; ++qt) {
                    float d[2][4];
                    tmem_ld_16x16(ta + 16 * qt, d);
                    if (qt == 3) {
                        tc_fence_before();
                        __syncwarp();
                        mbar_arrive_if(bar(BAR_F_EMPTY + tb), lane == 0);
                    }
#pragma unroll
                    for (int n = 0; n < 2; ++n) {
                        float (&sn)[4] = st[2 * qt + n];
                        const float2 a = mul2(add2(make_float2(sn[0], sn[1]), make_float2(d[n][0], d[n][1])), dlo2);
                        const float2 b = mul2(add2(make_float2(sn[2], sn[3]), make_float2(d[n][2], d[n][3])), dhi2);
                        sn[0] = a.x; sn[1] = a.y; sn[2] = b.x; sn[3] = b.y;
                    }
                }
            } else {
                // ---- decay too strong for one in-chunk reference point: the output warps run the exact fp32
                // recurrence over this chunk, token by token, on a copy of the state in shared memory.
                __syncwarp();
                mbar_arrive_if(bar(BAR_F_EMPTY + tb), lane == 0);
                // The copy lives in the pair of bf16 state operand tiles: this chunk's tile has no reader (its
                // products are skipped) and the other one is free once the products of chunk c-1 are done.
                // (The summary pass does not use these tiles at all.)
                if (!SUMMARY && c >= 1 && !mbar_wait(bar(BAR_B_DONE + (tb ^ 1)), ((c - 1) >> 1) & 1, abort_flag)) break;
                next_tile_free = true;
                // the fp32 copy overlays the bf16 rows of the other state warps: all of them have stored theirs first
                // (and the checkpoint copies that read those rows have left shared memory)
                if (CK_TMA && ck_on && lane == 0) bulk_wait_read<0>();
                __syncwarp();
                mbar_arrive_if(bar(BAR_SPRE), lane == 0);
                if (!mbar_wait(bar(BAR_SPRE), fb_uses & 1, abort_flag)) break;
                float* scr = reinterpret_cast<float*>(smem + OFF_SB);
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    *reinterpret_cast<float2*>(scr + c_lo * 64 + 8 * n + 2 * q) = make_float2(st[n][0], st[n][1]);
                    *reinterpret_cast<float2*>(scr + (c_lo + 8) * 64 + 8 * n + 2 * q) = make_float2(st[n][2], st[n][3]);
                }
                __syncwarp();
                mbar_arrive_if(bar(BAR_FB_READY), lane == 0);
                if (!mbar_wait(bar(BAR_FB_DONE), fb_uses & 1, abort_flag)) break;
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    const float2 lo = *reinterpret_cast<const float2*>(scr + c_lo * 64 + 8 * n + 2 * q);
                    const float2 hi = *reinterpret_cast<const float2*>(scr + (c_lo + 8) * 64 + 8 * n + 2 * q);
                    st[n][0] = lo.x; st[n][1] = lo.y; st[n][2] = hi.x; st[n][3] = hi.y;
                }
                // every state warp has re-read the copy before the operand tiles are rewritten
                __syncwarp();
                mbar_arrive_if(bar(BAR_SSYNC), lane == 0);
                if (!mbar_wait(bar(BAR_SSYNC), fb_uses & 1, abort_flag)) break;
                ++fb_uses;
            }
            if (!SUMMARY && !ck.last) {
                const int nb = tb ^ 1;
                if (!next_tile_free && !mbar_wait(bar(BAR_B_DONE + nb), ((c - 1) >> 1) & 1, abort_flag)) break;
                if (CKPT) {                          // the checkpoint copy of chunk c - 1 has finished reading this tile
                    if (lane == 0) bulk_wait_read<1>();
                    __syncwarp();
                }
                store_acc_bf16(sbase + OFF_SB + nb * TILE, 16 * sp, st, lane);
                fence_proxy_async();
                __syncwarp();
                mbar_arrive_if(bar(BAR_S_READY + nb), lane == 0);
                if (CKPT) ckpt_tile(nb, PERSIST ? (size_t)++pslot : ckpt_slot(seg * p.seg_chunks + c + 1));
            }
            if (SUMMARY && ck_on && ck.rem > 0) {    // (no product reads these tiles in a summary pass)
                const int nb = tb ^ 1;
                if (lane == 0) bulk_wait_read<1>();
                __syncwarp();
                store_acc_bf16(sbase + OFF_SB + nb * TILE, 16 * sp, st, lane);
                fence_proxy_async();
                __syncwarp();
                ckpt_tile(nb, ckpt_slot(seg * p.seg_chunks + c + 1));
            }
            if (PERSIST && ck.last && !lds32(abort_flag)) {
                if (BAL || p.state_out) store_state((size_t)ck.unit * 4096);
                if (CKPT && ck.rem == 0) store_ckpt(pslot + 1);
                if (BAL && ck.rem > 0) {             // a cut: the CTA that holds the rest of the unit may have the state
                    __threadfence();
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("st.release.gpu.global.u64 [%0], %1;"
                                     ::"l"(reinterpret_cast<unsigned long long*>(p.y + (size_t)(ck.row + L) * C + ck.h * 64) + sp), "l"(p.nonce) : "memory");
                }
            }
        }
        if (CK_TMA && ck_on && lane == 0) bulk_wait<0>();          // this warp's checkpoint copies have reached memory
        if (CKPT && !PERSIST && seg == p.nseg - 1 && !lds32(abort_flag)) store_ckpt(ckpt_slot(ckpt_chunks()));
        if (SUMMARY && p.ckpt) {
            if (seg == p.nseg - 1 && !lds32(abort_flag))     // the state after the last token
                store_ckpt(ckpt_slot(ckpt_chunks()));
        } else if (SUMMARY) {
            if (!lds32(abort_flag)) {
                float* sm = p.summaries + ((size_t)unit * (p.nseg - 1) + seg) * SUMMARY_FLOATS;
                if (trail_cut) dprod_lo = dprod_hi = 0.f;
                if (q == 0) { sm[c_lo] = dprod_lo; sm[c_lo + 8] = dprod_hi; }
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    *reinterpret_cast<float2*>(sm + 64 + c_lo * 64 + 8 * n + 2 * q) = make_float2(st[n][0], st[n][1]);
                    *reinterpret_cast<float2*>(sm + 64 + (c_lo + 8) * 64 + 8 * n + 2 * q) = make_float2(st[n][2], st[n][3]);
                }
            }
        } else if (!PERSIST && p.state_out && seg == p.nseg - 1 && !lds32(abort_flag)) {
            store_state(sb);
        } else if (TRAIL && seg < p.nseg - 1) {
            // a state that is no longer finite: marked in the segment's summary (see poison_later_segments; a later segment's CTA
            // that folds this summary meanwhile may see either)
            float z = 0.f;
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) z = fmaf(st[n][e], 0.f, z);
            if (z != 0.f) {
                float* sm = p.summaries + ((size_t)unit * (p.nseg - 1) + seg) * SUMMARY_FLOATS + 64;
#pragma unroll
                for (int n = 0; n < 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (st[n][e] * 0.f != 0.f) sm[(size_t)(e < 2 ? c_lo : c_lo + 8) * 64 + 8 * n + 2 * q + (e & 1)] = __int_as_float(0x7fc00000);
                sts32(sbase + OFF_MARK, 1u);
            }
        }
    } else if (warp < WARP_Y0) {
        // ============================== score warps ==============================
        const int sp = warp & 3;                 // rows t = 16*sp .. 16*sp+15 of the score block
        const int g = lane >> 2, q = lane & 3;
        for (int c = 0; PERSIST || c < (SUMMARY ? 0 : nchunks); ++c) {
            const int tb = c & 1, pt = (c >> 1) & 1, ppi = tb, sd = c & (NSIDE - 1);
            if (!mbar_wait(bar(BAR_F_FULL + tb), pt, abort_flag)) break;
            tc_fence_after();
            if (PERSIST && chunk_is_end(c)) {    // hand the end marker on, as above (after the products of chunk c-2)
                if (c >= NPP && !mbar_wait(bar(BAR_B_DONE + ppi), pt ^ 1, abort_flag)) break;
                __syncwarp();
                mbar_arrive_if(bar(BAR_PP_READY + ppi), lane == 0);
                break;
            }
            const bool safe = safe_at(sd);
            float d_lo = 0.f, d_hi = 0.f;
            if (safe && !C2) {
                const uint32_t du = sbase + OFF_DU + 4 * (sd * 64 + 16 * sp + g);
                d_lo = ldsf(du); d_hi = ldsf(du + 32);
            }
            if (c >= NPP && !mbar_wait(bar(BAR_B_DONE + ppi), pt ^ 1, abort_flag)) break;
            if (safe) {
                const uint32_t ta = tmem + ((uint32_t)(32 * sp) << 16) + TM_P + 64 * tb;
                const uint32_t tp = sbase + OFF_PP + ppi * TILE;
                float acc[4][4];
                tmem_ld_16x32(ta, acc);
                mask_scores_sp<0>(sp, acc, g, q, d_lo, d_hi);
                store_half_bf16<0>(tp, 16 * sp, acc, lane);
                tmem_ld_16x32(ta + 32, acc);
                tc_fence_before();
                __syncwarp();
                mbar_arrive_if(bar(BAR_F_EMPTY + tb), lane == 0);
                mask_scores_sp<1>(sp, acc, g, q, d_lo, d_hi);
                store_half_bf16<1>(tp, 16 * sp, acc, lane);
                fence_proxy_async();
            } else {
                __syncwarp();
                mbar_arrive_if(bar(BAR_F_EMPTY + tb), lane == 0);
            }
            __syncwarp();
            mbar_arrive_if(bar(BAR_PP_READY + ppi), lane == 0);
        }
    } else if (warp < WARP_E0) {
        // ============================== output warps ==============================
        const int sp = warp & 3;                 // rows t = 16*sp .. 16*sp+15 of the chunk
        const uint32_t slab = sbase + OFF_Y + sp * 2048;
        int fb_uses = 0;                         // chunks that took the token-by-token path so far
        if (SUMMARY) {
            // nothing to output: follow the chunks only to run the token-by-token path where one needs it
            for (int c = 0; c < nchunks; ++c) {
                const int tb = c & 1;
                if (!mbar_wait(bar(BAR_F_FULL + tb), (c >> 1) & 1, abort_flag)) break;
                if (!safe_at(c & (NSIDE - 1))) {
                    if (!mbar_wait(bar(BAR_FB_READY), fb_uses & 1, abort_flag)) break;
                    exact_chunk<false>(reinterpret_cast<float*>(smem + OFF_SB), p, h, sp, lane, row0 + (long long)c * L,
                                       min(L, len - c * L), C, col0);
                    __syncwarp();
                    mbar_arrive_if(bar(BAR_FB_DONE), lane == 0);
                    ++fb_uses;
                }
                __syncwarp();
                mbar_arrive_if(bar(BAR_F_EMPTY + tb), lane == 0);
            }
        }
        // Finch-C2 form: this warp's 16 rows of the second-value tensor come by TMA into a slab of its own,
        // one chunk ahead (requested as soon as the previous chunk's rows have been read out of it)
        const bool has_u2 = !SUMMARY && C2 && p.u2 != nullptr;
        const uint32_t u2slab = sbase + OFF_U2 + sp * 2048;
        bool u2_pending = false;                 // a slab copy is in flight; it completes the phase of parity u2_parity
        int u2_parity = 0, u2_loads = 0;         // (the slab's barrier completes one phase per load)
        // row: first row of the chunk whose 16 rows are wanted, in the unit with head column col; rem: chunks after it
        auto load_u2 = [&](int row, int col, int rem) {
            if (elect_one()) {
                mbar_expect_tx(bar(BAR_U2 + sp), 2048);
                tma_load_2d(u2slab, &tm_u2_16, col, row + 16 * sp, bar(BAR_U2 + sp));
                // the slab is single: pull the rows of the chunks after this one into L2 meanwhile, so that
                // their loads, which can only be issued once the slab is free, are short
                if (rem >= 2) tma_prefetch_2d(&tm_u2_16, col, row + 2 * L + 16 * sp);
                if (rem >= 3) tma_prefetch_2d(&tm_u2_16, col, row + 3 * L + 16 * sp);
            }
            __syncwarp();
            u2_pending = true;
            u2_parity = u2_loads & 1;
            ++u2_loads;
        };
        if (!PERSIST && !PAIR && has_u2 && nchunks > 0) load_u2((int)row0, col0, nchunks - 1);
        // Where a chunk's time does not hide that load (PAIR), two slabs per warp (by chunk parity), second-value rows in and y
        // rows out in their place, the load a chunk ahead and, in a stream, across units.  Balanced launches keep every SM
        // streaming (5 x 2011 tokens x 32 heads: 69.6 us with one slab, 62.3 with the pair); a training forward writes 16 KB
        // of state per chunk beside its y (4 x 16384 x 32 315.7 -> 295.6, 4 x 4096 93.3 -> 88.0, 8 x 2048 97.4 -> 93.6, 65536 x 32
        // in segments 381.9 -> 365.3, 8 x 1100 x 12 31.0 -> 30.9).  The plain prefill keeps one: with two, 8 x 4096 x 12
        // 80.0 -> 82.4, 8 x 1100 x 12 25.5 -> 27.0, 4 x 4096 x 32 85.2 -> 86.0, 4 x 16384 x 32 326.5 -> 324.8.
        int u2_issued = 0, u2_used = 0;          // one load per chunk: the i-th completes phase i / 2 of the barrier of slab i % 2
        auto u2_bar = [&](int i) { return bar(BAR_U2 + N_GW * (i & 1) + sp); };
        auto slab_of = [&](int i) { return (i & 1) ? u2slab : slab; };
        auto load_pair = [&](int row, int col, int rem) {
            if (elect_one()) {
                mbar_expect_tx(u2_bar(u2_issued), 2048);
                tma_load_2d(slab_of(u2_issued), &tm_u2_16, col, row + 16 * sp, u2_bar(u2_issued));
                if (rem >= 2) tma_prefetch_2d(&tm_u2_16, col, row + 2 * L + 16 * sp);
            }
            __syncwarp();
            ++u2_issued;
        };
        // the first chunk of the next unit of the stream, if there is one.  The producer is a ring ahead, so its descriptor
        // is there or about to be; it cannot be replaced before this warp has output the chunk.  (Not a wait on the
        // chunk's "full" barrier: this role lags behind it, and by more than one phase a parity means nothing.)
        auto load_pair_unit = [&](int c) -> bool {
            if (!__all_sync(0xffffffffu, desc_wait(sbase + OFF_DESC + 16 * (c & (NSIDE - 1)) + 4, ((c / NSIDE) & 1) * DESC_TAG, abort_flag))) return false;
            const Chunk nk = chunk_at(c);
            if (!nk.end) load_pair(nk.row, nk.h * 64, nk.rem);
            return true;
        };
        bool go = true;
        if (PAIR && PERSIST && has_u2) go = load_pair_unit(0);
        if (PAIR && !PERSIST && has_u2 && nchunks > 0) load_pair((int)row0, col0, nchunks - 1);
        for (int c = 0; (!PAIR || go) && (PERSIST || c < (SUMMARY ? 0 : nchunks)); ++c) {
            const int tb = c & 1;
            if (!mbar_wait(bar(BAR_B_DONE + tb), (c >> 1) & 1, abort_flag)) break;
            tc_fence_after();
            const Chunk ck = chunk_at(c);
            if (PERSIST && ck.end) break;
            const int ccol = PERSIST ? ck.h * 64 : col0;                  // this chunk's head column
            if (PERSIST && !PAIR && has_u2 && ck.first) load_u2(ck.row, ccol, ck.rem);   // (a unit's first slab is not fetched ahead)
            const bool safe = safe_at(c & (NSIDE - 1));
            if (lane == 0) bulk_wait_read<0>();   // this warp's previous store has finished reading its slab
            __syncwarp();
            if (PAIR && has_u2) {                 // ... which (chunk c - 1's) takes the rows of chunk c + 1
                if (!ck.last) load_pair(ck.row + L, ccol, ck.rem - 1);
                else if (PERSIST && !load_pair_unit(c + 1)) break;
            }
            const uint32_t out = PAIR ? slab_of(c) : slab;
            if (!safe) {
                // decay too strong for the tensor-core formulation: exact recurrence on the fp32 state copy
                // the state warps put in shared memory; writes this chunk's y rows itself
                mbar_arrive_if(bar(BAR_Y_EMPTY + tb), lane == 0);
                if (PAIR && has_u2) {             // keep the slab's phase in step
                    if (!mbar_wait(u2_bar(c), (c >> 1) & 1, abort_flag)) break;
                    ++u2_used;
                } else if (has_u2) {              // ... consume, then request the next
                    if (!mbar_wait(bar(BAR_U2 + sp), u2_parity, abort_flag)) break;
                    u2_pending = false;
                    if (!ck.last) load_u2(ck.row + L, ccol, ck.rem - 1);
                }
                if (!mbar_wait(bar(BAR_FB_READY), fb_uses & 1, abort_flag)) break;
                exact_chunk<true>(reinterpret_cast<float*>(smem + OFF_SB), p, ck.h, sp, lane, ck.row, ck.valid, C, ccol);
                __syncwarp();
                mbar_arrive_if(bar(BAR_FB_DONE), lane == 0);
                ++fb_uses;
                continue;
            }
            // ---- this warp's 16 rows of y -> bf16 slab -> global
            {
                const uint32_t ta = tmem + ((uint32_t)(32 * sp) << 16) + TM_Y + 64 * tb;
                float ya[4][4];
                tmem_ld_16x32(ta, ya);
                if (PAIR && has_u2) {
                    if (!mbar_wait(u2_bar(c), (c >> 1) & 1, abort_flag)) break;
                    ++u2_used;
                    add_slab_bf16<0>(ya, out, lane);
                } else if (has_u2) {
                    if (!mbar_wait(bar(BAR_U2 + sp), u2_parity, abort_flag)) break;
                    u2_pending = false;
                    add_slab_bf16<0>(ya, u2slab, lane);
                }
                store_half_bf16<0>(out, 0, ya, lane);
                tmem_ld_16x32(ta + 32, ya);
                tc_fence_before();
                __syncwarp();
                mbar_arrive_if(bar(BAR_Y_EMPTY + tb), lane == 0);
                if (has_u2) {
                    add_slab_bf16<1>(ya, PAIR ? out : u2slab, lane);
                    if (!PAIR) {
                        __syncwarp();
                        if (!ck.last) load_u2(ck.row + L, ccol, ck.rem - 1);
                    }
                }
                store_half_bf16<1>(out, 0, ya, lane);
            }
            fence_proxy_async();
            __syncwarp();
            const int rows = ck.valid - 16 * sp;
            const long long grow = (long long)ck.row + 16 * sp;
            if (rows >= 16) {
                if (lane == 0) {
                    tma_store_2d(&tm_y16, ccol, (int)grow, out);
                    bulk_commit();
                }
            } else {
                // ragged tail: the rows after `valid` belong to someone else, so copy row by row
                for (int i = lane; i < rows * 8; i += 32) {
                    const int t = i >> 3, ch = i & 7;
                    uint4 val;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(val.x), "=r"(val.y), "=r"(val.z), "=r"(val.w) : "r"(out + swz(t, ch << 4)));
                    *reinterpret_cast<uint4*>(p.y + (size_t)(grow + t) * C + ccol + ch * 8) = val;
                }
                __syncwarp();
            }
        }
        if (lane == 0) bulk_wait<0>();
        // leaving early (abort) with a slab copy still in flight: wait for it, it targets this CTA's memory
        if (u2_pending) mbar_wait(bar(BAR_U2 + sp), u2_parity, abort_flag, false);
        for (; PAIR && u2_used < u2_issued; ++u2_used) mbar_wait(u2_bar(u2_used), (u2_used >> 1) & 1, abort_flag, false);
    } else {
        // ============================== elementwise warps ==============================
        const int eset = (warp - WARP_E0) / N_EW;        // this set takes chunks eset, eset + 2, ...
        // tokens 8*tq .. 8*tq+7 of the chunk; the warp with the last tokens, which closes the chunk on top of its share,
        // is the set's first one and so sits on the scheduler (warp index mod 4) that holds no control warp
        const int tq = ((warp - WARP_E0) % N_EW + N_EW - 1) % N_EW;
        const int cq = lane & 15, th = lane >> 4;        // channels 4*cq .. 4*cq+3, tokens 8*tq + 4*th + (0..3)
        const int etid = tid - 32 * (WARP_E0 + eset * N_EW);   // 0..255 inside the set
        constexpr bool c2 = C2;                          // Finch-C2 form: keys times (1 - w), no bonus
        // (the bonus vector is only read where the bonus is computed: not in the Finch-C2 form, not in a summary pass)
        const float4 u4 = (c2 || SUMMARY || PERSIST) ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4*>(p.u + h * 64 + 4 * cq);
        float2 ua = make_float2(u4.x, u4.y), ub = make_float2(u4.z, u4.w);
        int u_head = -1;                                 // persistent launches: the head whose bonus vector ua, ub hold
        uint32_t roff[4];                                // swizzled byte offsets of this lane's 8 bytes in its 4 rows
#pragma unroll
        for (int tt = 0; tt < 4; ++tt) roff[tt] = swz(8 * tq + 4 * th + tt, 8 * cq);
        const float2 kLog2e = make_float2(LOG2E, LOG2E), kLogLog = make_float2(LOG2_LOG2E, LOG2_LOG2E);
        int s = STAGE_STEP * eset, ph = 0;               // ring stage of this set's current chunk and its "full" barrier's phase bit
        for (int c = eset; PERSIST || c < nchunks; c += N_ESET) {
            const int sd = c & (NSIDE - 1);
            const uint32_t tx = sbase + OFF_RING + s * STAGE, tv = tx + 3 * TILE;
            uint32_t ax[4];                              // this lane's 8 bytes in its 4 rows of the x tile; r at +TILE, k at +2 TILE
#pragma unroll
            for (int tt = 0; tt < 4; ++tt) ax[tt] = tx + roff[tt];
            // (c & 1 is eset: the one that leaves fewer spills in the variant)
            if (!mbar_wait(bar(BAR_FULL_RKV + (TRAIL || SUMMARY ? eset : c & 1) * NS + s), ph, abort_flag)) break;
            Chunk ck;                                    // (this role needs the valid-token count, the head and the end flag only)
            if constexpr (PERSIST) {
                const uint32_t meta = lds32(sbase + OFF_DESC + 16 * (c & (NSIDE - 1)) + 4);
                ck.valid = (int)(meta & 0xff); ck.h = (int)(meta >> 16); ck.end = (meta & DESC_END) != 0;
            } else {
                ck.valid = min(L, len - c * L); ck.h = h; ck.end = false;
            }
            if (PERSIST && ck.end) {                     // hand the end marker to the issuer of the input-only products
                __syncwarp();
                mbar_arrive_if(bar(BAR_RK_READY + s), lane == 0);
                break;
            }
            if (PERSIST && !c2 && ck.h != u_head) {      // the stream moved on to another head: its bonus vector
                const float4 un = *reinterpret_cast<const float4*>(p.u + ck.h * 64 + 4 * cq);
                ua = make_float2(un.x, un.y); ub = make_float2(un.z, un.w);
                u_head = ck.h;
            }
            if (ck.valid < L) {
                // Ragged last chunk: rows past the end of the sequence hold another sequence's tokens (or the
                // out-of-range fill).  Each lane rewrites its own part of those rows before it reads them
                // back: x = -inf (no decay), r = k = 0; the v rows are zeroed for the tensor core.
                const int valid = ck.valid;
#pragma unroll
                for (int tt = 0; tt < 4; ++tt)
                    if (8 * tq + 4 * th + tt >= valid) {
                        sts64(ax[tt], make_uint2(0xff80ff80u, 0xff80ff80u));
                        if (!SUMMARY) sts64_at<TILE>(ax[tt], make_uint2(0u, 0u));
                        sts64_at<2 * TILE>(ax[tt], make_uint2(0u, 0u));
                    }
                for (int i = etid; i < (L - valid) * 8; i += 32 * N_EW)
                    sts128z(tv + (valid + (i >> 3)) * 128 + ((i & 7) << 4));
            }
            // ---- phase A: log2-decay magnitudes e = exp(x) log2(e), inclusive cumulative sums over this lane's tokens
            float2 aa[4], ab[4];                         // -(cumulative e): channel pairs (0,1) and (2,3)
            {
                uint2 xw[4];
#pragma unroll
                for (int tt = 0; tt < 4; ++tt) xw[tt] = lds64(ax[tt]);
                float2 ra = make_float2(0.f, 0.f), rb = ra;
#pragma unroll
                for (int tt = 0; tt < 4; ++tt) {
                    const float2 ea = ex2_2(fma2(bf_pair(xw[tt].x), kLog2e, kLogLog));
                    const float2 eb = ex2_2(fma2(bf_pair(xw[tt].y), kLog2e, kLogLog));
                    ra = sub2(ra, ea); rb = sub2(rb, eb);
                    aa[tt] = ra; ab[tt] = rb;
                }
            }
            // the other half-warp's total: lanes th = 1 start after it, lanes th = 0 add it to form the warp's total
            float2 oa, ob;
            oa.x = __shfl_xor_sync(0xffffffffu, aa[3].x, 16); oa.y = __shfl_xor_sync(0xffffffffu, aa[3].y, 16);
            ob.x = __shfl_xor_sync(0xffffffffu, ab[3].x, 16); ob.y = __shfl_xor_sync(0xffffffffu, ab[3].y, 16);
            const uint32_t totc = sbase + OFF_TOT + 4 * ((c % NTOT) * N_EW * 64 + 4 * cq);
            {
                const float2 wa = add2(aa[3], oa), wb = add2(ab[3], ob);
                stsf4_if(totc + 256 * tq, make_float4(wa.x, wa.y, wb.x, wb.y), th == 0);
                if (th == 0) { oa = make_float2(0.f, 0.f); ob = oa; }
            }
            __syncwarp();
            mbar_arrive_if(bar(BAR_ESYNC + eset), lane == 0);
            if (!mbar_wait(bar(BAR_ESYNC + eset), (c >> 1) & 1, abort_flag)) break;
            // cumulative sum at the end of the warps before this one: their totals, fetched together and added as a tree
            switch (tq) {
            case 1: add_totals<1>(totc, oa, ob); break;
            case 2: add_totals<2>(totc, oa, ob); break;
            case 3: add_totals<3>(totc, oa, ob); break;
            case 4: add_totals<4>(totc, oa, ob); break;
            case 5: add_totals<5>(totc, oa, ob); break;
            case 6: add_totals<6>(totc, oa, ob); break;
            case 7: add_totals<7>(totc, oa, ob); break;
            default: break;
            }
            // ---- phase B, in place: r -> R^ = r 2^{a_{t-1}}, k -> K^ = k 2^{-a_t}; bonus partials
            uint2 rw[4], kw[4];
#pragma unroll
            for (int tt = 0; tt < 4; ++tt) {             // all loads first: they are ordered with the stores below
                if (!SUMMARY) rw[tt] = lds64_at<TILE>(ax[tt]);
                kw[tt] = lds64_at<2 * TILE>(ax[tt]);
            }
            float du[4];
            float2 pa = oa, pb = ob;                     // a_{t-1}
            // Finch-C2: k (1 - w_t) 2^{-a_t} = k (2^{-a_t} - 2^{-a_{t-1}}) since w_t 2^{-a_t} = 2^{-a_{t-1}}:
            // the previous token's key scale is subtracted (no further exponential but the run's first)
            float2 qa = make_float2(0.f, 0.f), qb = qa;
            if (c2) { qa = ex2_2(make_float2(-oa.x, -oa.y)); qb = ex2_2(make_float2(-ob.x, -ob.y)); }
#pragma unroll
            for (int tt = 0; tt < 4; ++tt) {
                const float2 ca = add2(oa, aa[tt]), cb = add2(ob, ab[tt]);     // a_t
                const float2 ska = ex2_2(make_float2(-ca.x, -ca.y)), skb = ex2_2(make_float2(-cb.x, -cb.y));
                const float2 k0 = bf_pair(kw[tt].x), k1 = bf_pair(kw[tt].y);
                const float2 kh0 = mul2(k0, c2 ? sub2(ska, qa) : ska), kh1 = mul2(k1, c2 ? sub2(skb, qb) : skb);
                qa = ska; qb = skb;
                kw[tt] = make_uint2(pack_bf16(kh0.x, kh0.y), pack_bf16(kh1.x, kh1.y));
                if (!SUMMARY) {
                    const float2 sra = ex2_2(pa), srb = ex2_2(pb);
                    const float2 r0 = bf_pair(rw[tt].x), r1 = bf_pair(rw[tt].y);
                    const float2 rh0 = mul2(r0, sra), rh1 = mul2(r1, srb);
                    rw[tt] = make_uint2(pack_bf16(rh0.x, rh0.y), pack_bf16(rh1.x, rh1.y));
                    if (!C2) {
                        const float2 acc = fma2(mul2(r1, k1), ub, mul2(mul2(r0, k0), ua));
                        du[tt] = acc.x + acc.y;
                    }
                }
                pa = ca; pb = cb;
            }
#pragma unroll
            for (int tt = 0; tt < 4; ++tt) {
                if (!SUMMARY) sts64_at<TILE>(ax[tt], rw[tt]);
                sts64_at<2 * TILE>(ax[tt], kw[tt]);
            }
            // reduce the 4 bonus partials over the 16 lanes of a half-warp (transposing butterfly):
            // lanes with bits (3,2) = (b8, b4) end with token 2*b8 + b4
            if (!SUMMARY && !C2) {                       // (the Finch-C2 form has no bonus: the diagonal of P' is zero)
                const bool b8 = lane & 8, b4 = lane & 4;
                float w2[2], w1;
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float send = b8 ? du[m] : du[m + 2], keep = b8 ? du[m + 2] : du[m];
                    w2[m] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
                }
                {
                    const float send = b4 ? w2[0] : w2[1], keep = b4 ? w2[1] : w2[0];
                    w1 = keep + __shfl_xor_sync(0xffffffffu, send, 4);
                }
                w1 += __shfl_xor_sync(0xffffffffu, w1, 2);
                w1 += __shfl_xor_sync(0xffffffffu, w1, 1);
                stsf_if(sbase + OFF_DU + 4 * (sd * 64 + 8 * tq + (lane >> 2)), w1, (lane & 3) == 0);
            }
            if (tq == N_EW - 1) {
                // pa, pb now hold a_L on the lanes that own the chunk's last tokens (th = 1)
                bool ok = true;
                if (th == 1) {
                    const float2 da = ex2_2(pa), db = ex2_2(pb);
                    stsf4(sbase + OFF_DL + 4 * (sd * 64 + 4 * cq), make_float4(da.x, da.y, db.x, db.y));
                    ok = (pa.x >= -A2_MAX) && (pa.y >= -A2_MAX) && (pb.x >= -A2_MAX) && (pb.y >= -A2_MAX);   // false for NaN as well
                }
                const bool all_ok = __all_sync(0xffffffffu, ok);
                if (lane == 0) sts32(sbase + OFF_SAFE + 4 * sd, all_ok ? 1u : 0u);
            }
            fence_proxy_async();                  // the scaled tiles are read by the tensor core (async proxy)
            __syncwarp();
            mbar_arrive_if(bar(BAR_RK_READY + s), lane == 0);
            if (++s == NS) { s = 0; ph ^= 1; }
        }
    }

    // every role is done with tensor memory (or the CTA is aborting): release it
    tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA_F) {
        tc_fence_after();
        tmem_dealloc(tmem, TM_COLS);
    }
    if (TRAIL)
        poison_later_segments<CKPT>(p, unit, seg, lds32(sbase + OFF_MARK) != 0, reinterpret_cast<int*>(smem + OFF_TOT),
                                    reinterpret_cast<int*>(smem + OFF_TOT) + 64, CKPT ? ckpt_slot(0) : 0);
}

// One warp that waits, with the kernel's own bounded wait, on a barrier nobody arrives on: the wait runs out after
// limit_us microseconds, raises the status flag and the kernel returns.  (Exercises the time-out path of the waits
// above without disturbing anything: see gf_wkv6_selftest_wait_timeout.)
__global__ void __launch_bounds__(32) wait_timeout_selftest_kernel(uint32_t limit_us)
{
    __shared__ __align__(8) unsigned long long words[2];       // {abort word, limit}, mbarrier
    const uint32_t abort_flag = smem_u32(&words[0]), bar = smem_u32(&words[1]);
    if (threadIdx.x == 0) {
        sts32(abort_flag, 0u);
        sts32(abort_flag + 4, limit_us);
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    mbar_wait_warp(bar, 0, abort_flag);
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// [rows][C] bf16 tensor, box = box_rows rows x 64 channels (128 bytes), 128-byte swizzle
inline bool make_map(CUtensorMap* tm, const void* base, long long rows, long long C, int box_rows,
                     CUtensorMapL2promotion promotion = CU_TENSOR_MAP_L2_PROMOTION_L2_256B)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)C * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, promotion,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace ck

// Chooses the sequence split of a call: with fewer (sequence, head) units than half the SMs, each
// sequence is cut into up to 8 segments of at least 8 chunks so that the grid fills the GPU (T: the
// sequence length, for a packed call the longest one).  Returns the number of segments (1: no split) and
// sets seg_chunks; summary_bytes is the scratch the split uses: per unit one summary for every segment but
// the last and a copy of the start state.  cap_bytes bounds that scratch: the split takes the largest
// segment count that fits (1 if not even two segments do).
constexpr size_t STATE_FLOATS = 64 * 64;
inline size_t split_scratch_bytes(long long units, int nseg)
{
    return (size_t)units * ((size_t)(nseg - 1) * ck::SUMMARY_FLOATS + STATE_FLOATS) * sizeof(float);
}
inline int choose_split(long long units, int T, int n_sm, int* seg_chunks, size_t* summary_bytes,
                        size_t cap_bytes = ~(size_t)0)
{
    *seg_chunks = 0;
    *summary_bytes = 0;
    const int nchunks = (T + ck::L - 1) / ck::L;
    if (units <= 0 || n_sm <= 0 || units * 2 > n_sm) return 1;
    int want = (int)(n_sm / units);
    if (want > 8) want = 8;
    if (want > nchunks / 8) want = nchunks / 8;
    for (; want >= 2; --want) {
        const int sc = (nchunks + want - 1) / want;
        const int g = (nchunks + sc - 1) / sc;
        if (g < 2) return 1;
        const size_t bytes = split_scratch_bytes(units, g);
        if (bytes > cap_bytes) continue;
        *seg_chunks = sc;
        *summary_bytes = bytes;
        return g;
    }
    return 1;
}

// Opts the instantiations of the chunked kernel in to their dynamic shared-memory size, once per device.
inline bool chunked_kernel_attributes()
{
    static PerDeviceFlag attr_set;                   // zero-initialised
    const int dev = current_device();
    if (dev < 0) return false;
    if (!attr_set.is_set(dev)) {
        if (cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, 0, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, 0, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, 0, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, 0, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, false, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess ||
            cudaFuncSetAttribute(ck::wkv6_chunked_kernel<false, true, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM_ALLOC) != cudaSuccess)
            return false;
        attr_set.set(dev);
    }
    return true;
}

// Prepares the scratch of a packed persistent launch: zeroes the unit counter and, for up to ORDER_MAX_SEQ
// sequences, writes the sequence indices by decreasing length (rank by counting; ties by index).
constexpr int ORDER_MAX_SEQ = 8192;
constexpr size_t ORDER_OFFSET = 64;                  // bytes from the counter to the order array
__global__ void __launch_bounds__(1024)
wkv6_order_kernel(const int32_t* __restrict__ cu, int S, unsigned int* counter, int32_t* order)
{
    __shared__ int len[ORDER_MAX_SEQ];
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
    if (threadIdx.x == 0) *counter = 0u;
    if (!order) return;
    for (int i = threadIdx.x; i < S; i += blockDim.x) len[i] = cu[i + 1] - cu[i];
    __syncthreads();
    for (int i = threadIdx.x; i < S; i += blockDim.x) {
        const int li = len[i];
        int rank = 0;
        for (int j = 0; j < S; ++j) rank += (len[j] > li) || (len[j] == li && j < i);
        order[rank] = i;
    }
}

// Scratch a packed call with more units than SMs uses: the counter and the order array.
inline size_t persistent_scratch_bytes(int n_seq)
{
    return ORDER_OFFSET + (n_seq <= ORDER_MAX_SEQ ? (size_t)n_seq * sizeof(int32_t) : 0);
}

// Launches the chunked kernel.  Dense: cu == nullptr, n_seq = B, T = sequence length.
// Packed: cu = device cu_seqlens, n_seq = S, T = max_seqlen.  total_rows = rows of the [rows][H*64] tensors.
// scratch / scratch_bytes: optional device memory for the sequence split (see choose_split); without
// enough of it the call runs unsplit.
// limit of the device-side waits of the launches below, in microseconds (0: default); set by gf_wkv6_set_wait_limit
inline std::atomic<uint32_t>& wait_limit_us()
{
    static std::atomic<uint32_t> v{0};
    return v;
}

// A number no earlier launch of this process has used, and that memory left by anything else does not hold (from the time the
// first one was drawn; not from std::random_device, which may throw, and nothing may be thrown through the C interface).
inline unsigned long long launch_nonce()
{
    static std::atomic<unsigned long long> next{(unsigned long long)std::chrono::system_clock::now().time_since_epoch().count()};
    unsigned long long z = next.fetch_add(0x9e3779b97f4a7c15ull, std::memory_order_relaxed);     // (Weyl sequence, then a bijective mix)
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Whether cutting units between CTAs (Params::bal_chunks) shortens a dense launch of more units than SMs: whole units end
// with a round that not every SM has one for.  The cut itself costs about two chunk times (its chunk enters the stream like
// a unit's first one), and while all SMs stream, a chunk takes a fifth longer than with the SMs of a last round idle; so
// it is taken where it saves more than four chunk times and more than a fifth of the launch.  Measured (us, whole units ->
// balanced): 160 units of 128 chunks 258 -> 163, of 20 chunks 53 -> 39; 156 of 39 chunks 93 -> 61; 192 of 63 chunks
// 135 -> 106; 320 of 47 chunks 159 -> 130; not taken: 256 of 32 chunks 79.7 -> 80.5.
inline bool balance_pays(long long units, int n_chunks, int n_sm)
{
    const long long rounds = (units + n_sm - 1) / n_sm, idle = rounds * n_sm - units;
    return idle * n_chunks > 4LL * n_sm && idle * 5 > rounds * n_sm && 2LL * n_sm * n_sm * n_chunks < (1LL << 32);   // (32-bit ranges)
}

// Launches a persistent instantiation with one CTA per SM; cooperative if its CTAs wait for one another.
template <typename Kernel>
inline cudaError_t launch_persistent(Kernel kernel, int n_sm, bool cooperative, cudaStream_t st, const CUtensorMap& tr, const CUtensorMap& tk,
                                     const CUtensorMap& tv, const CUtensorMap& tx, const CUtensorMap& ty, const CUtensorMap& tu2,
                                     const ck::Params& p, const CUtensorMap& tck)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_sm);
    cfg.blockDim = dim3(ck::THREADS);
    cfg.dynamicSmemBytes = ck::SMEM_ALLOC;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cooperative ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, tr, tk, tv, tx, ty, tu2, p, tck);
}

inline gf_status_t chunked_prefill(const __nv_bfloat16* r, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                   const __nv_bfloat16* x, const float* u, const float* state_in, float* state_out,
                                   __nv_bfloat16* y, const int32_t* cu, int n_seq, int T, long long total_rows, int H,
                                   cudaStream_t st, std::atomic<uint64_t>* launches, float* scratch = nullptr,
                                   size_t scratch_bytes = 0, const __nv_bfloat16* u2 = nullptr, int c2 = 0,
                                   float* ckpt = nullptr)
{
    const long long units = (long long)n_seq * H;
    if (units <= 0 || units > 0x7fffffffLL || total_rows <= 0) return GF_ERR_INVALID_ARG;
    // what this kernel cannot take (32-bit TMA row coordinates with a chunk of slack; no tensor-map encoder in the
    // driver) is reported as unsupported, so that the caller can run the token-by-token kernel instead
    if (total_rows >= (1LL << 31) - 64 || !ck::encode_fn()) return GF_ERR_UNSUPPORTED;
    if (!chunked_kernel_attributes()) return GF_ERR_CUDA;
    CUtensorMap tr, tk, tv, tx, ty, tu2;
    const long long C = (long long)H * 64;
    if (!ck::make_map(&tr, r, total_rows, C, 64) || !ck::make_map(&tk, k, total_rows, C, 64) ||
        !ck::make_map(&tv, v, total_rows, C, 64) || !ck::make_map(&tx, x, total_rows, C, 64) ||
        !ck::make_map(&ty, y, total_rows, C, 16) || !ck::make_map(&tu2, u2 ? (const void*)u2 : (const void*)y, total_rows, C, 16))
        return GF_ERR_CUDA;
    int seg_chunks = 0, nseg = 1;
    if (scratch && !(ckpt && cu)) {                           // packed calls split by max_seqlen: segments past a sequence's end are empty
        size_t need = 0;
        nseg = choose_split(units, T, sm_count(), &seg_chunks, &need, scratch_bytes);   // (never splits with more units than half the SMs)
        if (nseg > 1 && units * nseg > 0x7fffffffLL) nseg = 1;
    }
    ck::Params p{r, k, v, x, y, u, state_in, state_out, cu, T, H, scratch, seg_chunks, nseg, u2, c2};
    CUtensorMap tck = ty;                            // (read only by the launches that keep checkpoints)
    if (nseg > 1 && state_in) p.state_copy = scratch + (size_t)units * (nseg - 1) * ck::SUMMARY_FLOATS;
    // A late start (Params::trail) runs about 42 chunks of a segment at the decays of a trained model (w in [0.69, 0.998]), and
    // costs 5 to 10 us of looking and marking where the decays are too slow for one: it is allowed where segments are long enough
    // to gain more than that.  (us without -> with a late start at such decays / at slow ones; 32 units of 4 segments of 48 chunks
    // 91 -> 107 / 91 -> 99, of 64 115 -> 124 / 115 -> 123, of 96 163 -> 155 / 163 -> 171, of 128 218 -> 189 / 218 -> 222, of 192
    // 317 -> 261 / 320 -> 332, of 512 847 -> 596 / 900 -> 910; 8 units of 8 segments of 96 160 -> 153 / 160 -> 168, of 128
    // 206 -> 181 / 206 -> 215.)
    p.trail = nseg > 1 && seg_chunks >= 128;
    p.wait_limit_us = wait_limit_us().load(std::memory_order_relaxed);
    if (ckpt) {
        // a training step's forward pass: one CTA per unit and segment, the chunk-start states kept for the gradient
        p.ckpt_slots = cu ? total_rows / ck::L + 2LL * n_seq : 0;
        const long long n_ckpt = cu ? (long long)H * p.ckpt_slots : units * ((T + ck::L - 1) / ck::L + 1);
        if (n_ckpt * 64 >= (1LL << 31)) return GF_ERR_UNSUPPORTED;
        if (!ck::make_map(&tck, ckpt, n_ckpt * 64, 64, 16)) return GF_ERR_CUDA;      // the checkpoints as [slots * 64][64] bf16
        if (nseg > 1) {
            if (c2) ck::wkv6_chunked_kernel<true, true><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tr, tk, tv, tx, ty, tu2, p, tck);
            else ck::wkv6_chunked_kernel<true, false><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tr, tk, tv, tx, ty, tu2, p, tck);
            launches->fetch_add(1, std::memory_order_relaxed);
            if (cudaGetLastError() != cudaSuccess) return GF_ERR_CUDA;
        }
        p.ckpt = ckpt;
        const int n_sm_ck = sm_count(), unit_chunks = (T + ck::L - 1) / ck::L;
        if (!cu && nseg == 1 && state_out && n_sm_ck > 0 && units > n_sm_ck && balance_pays(units, unit_chunks, n_sm_ck)) {
            p.n_units = (int)units;                  // a balanced stream per SM (see below)
            p.bal_chunks = unit_chunks;
            p.nonce = launch_nonce();
            const cudaError_t e = c2 ? launch_persistent(ck::wkv6_chunked_kernel<false, true, 2, true>, n_sm_ck, true, st, tr, tk, tv, tx, ty, tu2, p, tck)
                                     : launch_persistent(ck::wkv6_chunked_kernel<false, false, 2, true>, n_sm_ck, true, st, tr, tk, tv, tx, ty, tu2, p, tck);
            if (e != cudaErrorCooperativeLaunchTooLarge) {
                launches->fetch_add(1, std::memory_order_relaxed);
                return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
            }
            cudaGetLastError();                      // (fewer SMs to be had than the device has: whole units below)
            p.bal_chunks = 0;
        }
        if (nseg == 1 && n_sm_ck > 0 && units > n_sm_ck && H <= ck::STREAM_MAX_HEADS &&
            (cu ? units >= 6LL * n_sm_ck || (unit_chunks <= 48 && units >= 3LL * n_sm_ck) : unit_chunks <= 32 && units >= 3LL * n_sm_ck) &&
            (!cu || (scratch && scratch_bytes >= persistent_scratch_bytes(n_seq)))) {
            // A stream of whole units per SM; packed: the longest sequences first, as in the prefill without checkpoints.
            // Dense (us, one CTA per unit -> stream, classic; Finch-C2): 448 units of 8..64 chunks the same; 576 of 8 chunks 69 ->
            // 57; 82 -> 65, of 16 105 -> 98; 124 -> 111, of 32 179 -> 182; 209 -> 204, of 48 257 -> 262; 288 -> 301, of 64
            // 334 -> 347; 372 -> 392; 896 of 32 312 -> 319; 349 -> 347, of 48 430 -> 466; 469 -> 498; 1184 of 32 348 -> 346;
            // 395 -> 396, of 48 508 -> 510; 560 -> 606: up to 32 chunks.
            // Packed, where a stream also hands out the longest first: 768 units of up to 14 chunks 96 -> 84 us, 45 175 -> 150, 89
            // 380 -> 365 (all long, 32..47: 290 -> 298); 1280 of up to 63 409 -> 392; 2048 of up to 64 657 -> 671 (Finch-C2
            // 755 -> 750).
            p.n_units = (int)units;
            if (cu) {
                p.ticket = reinterpret_cast<unsigned int*>(scratch);
                int32_t* order = n_seq <= ORDER_MAX_SEQ ? reinterpret_cast<int32_t*>(reinterpret_cast<char*>(scratch) + ORDER_OFFSET) : nullptr;
                p.order = order;
                const cudaError_t eo = launch_pdl(wkv6_order_kernel, 1, 1024, 0, st, cu, n_seq, p.ticket, order);
                launches->fetch_add(1, std::memory_order_relaxed);
                if (eo != cudaSuccess) return GF_ERR_CUDA;
            }
            const cudaError_t e = c2 ? launch_persistent(ck::wkv6_chunked_kernel<false, true, 1, true>, n_sm_ck, false, st, tr, tk, tv, tx, ty, tu2, p, tck)
                                     : launch_persistent(ck::wkv6_chunked_kernel<false, false, 1, true>, n_sm_ck, false, st, tr, tk, tv, tx, ty, tu2, p, tck);
            launches->fetch_add(1, std::memory_order_relaxed);
            return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
        }
        const auto kernel = p.trail ? (c2 ? ck::wkv6_chunked_kernel<false, true, 0, true, true> : ck::wkv6_chunked_kernel<false, false, 0, true, true>)
                                    : (c2 ? ck::wkv6_chunked_kernel<false, true, 0, true> : ck::wkv6_chunked_kernel<false, false, 0, true>);
        kernel<<<(unsigned)(units * nseg), ck::THREADS, ck::SMEM_ALLOC, st>>>(tr, tk, tv, tx, ty, tu2, p, tck);
        launches->fetch_add(1, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess ? GF_OK : GF_ERR_CUDA;
    }
    const int n_sm = sm_count();
    // More units than SMs: one CTA per SM walks a stream of units, so that a unit's pipeline fill overlaps the
    // drain of the one before it.  That saves about 4.5 us per unit and costs about 3 % more instructions per
    // chunk (descriptor reads), so it is taken for short units or many units per SM (measured: 512 units of 64
    // chunks lose 3 %, 1184 units of 32 chunks gain 2 %, 4096 units of 8 chunks gain 30 %).  Packed calls draw
    // their units from a counter in the scratch (their lengths differ); dense calls take every gridDim-th unit
    // (drawing them from the counter too was measured 3 % slower).
    const int max_chunks = (T + ck::L - 1) / ck::L;
    // Where whole units would leave SMs idle in the last round, dense calls cut units between CTAs (balance_pays).
    if (!cu && state_out && nseg == 1 && n_sm > 0 && units > n_sm && balance_pays(units, max_chunks, n_sm)) {
        p.n_units = (int)units;
        p.bal_chunks = max_chunks;
        p.nonce = launch_nonce();
        const cudaError_t e = c2 ? launch_persistent(ck::wkv6_chunked_kernel<false, true, 2>, n_sm, true, st, tr, tk, tv, tx, ty, tu2, p, tck)
                                 : launch_persistent(ck::wkv6_chunked_kernel<false, false, 2>, n_sm, true, st, tr, tk, tv, tx, ty, tu2, p, tck);
        if (e != cudaErrorCooperativeLaunchTooLarge) {
            launches->fetch_add(1, std::memory_order_relaxed);
            return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
        }
        cudaGetLastError();                          // (fewer SMs to be had than the device has: whole units below)
        p.bal_chunks = 0;
    }
    if (nseg == 1 && n_sm > 0 && units > n_sm && H <= ck::STREAM_MAX_HEADS && (units >= 6LL * n_sm || max_chunks <= 48) &&
        (!cu || (scratch && scratch_bytes >= sizeof(unsigned int)))) {
        p.n_units = (int)units;
        if (cu) {
            p.ticket = reinterpret_cast<unsigned int*>(scratch);
            int32_t* order = nullptr;
            if (n_seq <= ORDER_MAX_SEQ && scratch_bytes >= persistent_scratch_bytes(n_seq))
                order = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(scratch) + ORDER_OFFSET);
            p.order = order;
            const cudaError_t eo = launch_pdl(wkv6_order_kernel, 1, 1024, 0, st, cu, n_seq, p.ticket, order);
            launches->fetch_add(1, std::memory_order_relaxed);
            if (eo != cudaSuccess) return GF_ERR_CUDA;
        }
        const cudaError_t e = launch_pdl(c2 ? ck::wkv6_chunked_kernel<false, true, 1> : ck::wkv6_chunked_kernel<false, false, 1>, (unsigned)n_sm,
                                         ck::THREADS, ck::SMEM_ALLOC, st, tr, tk, tv, tx, ty, tu2, p, tck);
        launches->fetch_add(1, std::memory_order_relaxed);
        return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
    }
    if (nseg > 1) {
        if (c2) ck::wkv6_chunked_kernel<true, true><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tr, tk, tv, tx, ty, tu2, p, tck);
        else ck::wkv6_chunked_kernel<true, false><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tr, tk, tv, tx, ty, tu2, p, tck);
        launches->fetch_add(1, std::memory_order_relaxed);
        if (cudaGetLastError() != cudaSuccess) return GF_ERR_CUDA;
    }
    if (nseg > 1) {
        // behind the summary launch: may start before it has finished (see the top of the kernel)
        const auto kernel = p.trail ? (c2 ? ck::wkv6_chunked_kernel<false, true, 0, false, true> : ck::wkv6_chunked_kernel<false, false, 0, false, true>)
                                    : (c2 ? ck::wkv6_chunked_kernel<false, true> : ck::wkv6_chunked_kernel<false, false>);
        const cudaError_t e = launch_pdl(kernel, (unsigned)(units * nseg), ck::THREADS, ck::SMEM_ALLOC, st, tr, tk, tv, tx, ty, tu2, p, tck);
        launches->fetch_add(1, std::memory_order_relaxed);
        return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
    }
    const cudaError_t e = launch_pdl(c2 ? ck::wkv6_chunked_kernel<false, true> : ck::wkv6_chunked_kernel<false, false>, (unsigned)units, ck::THREADS,
                                     ck::SMEM_ALLOC, st, tr, tk, tv, tx, ty, tu2, p, tck);
    launches->fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
}

// Summary of whole sequences (the pair of the affine map S -> diag(D) S + dS that a sequence applies to
// the state): one summary launch with a single segment per unit.  summary: [n_seq*H][64 + 64*64] fp32.
inline gf_status_t chunked_summary(const __nv_bfloat16* k, const __nv_bfloat16* v, const __nv_bfloat16* x, float* summary,
                                   int n_seq, int T, int H, int c2, cudaStream_t st, std::atomic<uint64_t>* launches)
{
    const long long units = (long long)n_seq * H, total_rows = (long long)n_seq * T;
    if (units <= 0 || units > 0x7fffffffLL || total_rows <= 0 || total_rows >= (1LL << 31) - 64) return GF_ERR_INVALID_ARG;
    if (!chunked_kernel_attributes()) return GF_ERR_CUDA;
    CUtensorMap tk, tv, tx, tdummy;
    const long long C = (long long)H * 64;
    if (!ck::make_map(&tk, k, total_rows, C, 64) || !ck::make_map(&tv, v, total_rows, C, 64) ||
        !ck::make_map(&tx, x, total_rows, C, 64) || !ck::make_map(&tdummy, k, total_rows, C, 16))
        return GF_ERR_CUDA;
    // two nominal segments of which the first covers the whole sequence: the summary launch handles
    // every segment but the last
    ck::Params p{nullptr, k, v, x, nullptr, nullptr, nullptr, nullptr, nullptr, T, H, summary, (T + ck::L - 1) / ck::L, 2, nullptr, c2};
    const CUtensorMap tck = tdummy;
    p.wait_limit_us = wait_limit_us().load(std::memory_order_relaxed);
    if (c2) ck::wkv6_chunked_kernel<true, true><<<(unsigned)units, ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
    else ck::wkv6_chunked_kernel<true, false><<<(unsigned)units, ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
    launches->fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? GF_OK : GF_ERR_CUDA;
}

// Checkpoint pass of dense sequences: the state before every chunk of 64 tokens and after the last one,
// ckpt [n_seq*H][chunks + 1][64][64] bf16, from state_in (NULL: zero).  One summary-variant launch (state only: reads
// k, v and the decay logits); with `summaries` (scratch of units x (nseg - 1) summaries) and nseg > 1 two: the sequences
// split into segments as in a split prefill call.
inline gf_status_t chunked_checkpoints(const __nv_bfloat16* k, const __nv_bfloat16* v, const __nv_bfloat16* x,
                                       const float* state_in, float* ckpt, int n_seq, int T, int H, cudaStream_t st,
                                       std::atomic<uint64_t>* launches, int c2 = 0, float* summaries = nullptr,
                                       int nseg = 1, int seg_chunks = 0, const int32_t* cu = nullptr,
                                       long long packed_rows = 0)
{
    // packed sequences (cu: device cu_seqlens of n_seq sequences over packed_rows rows, T = max_seqlen): split by
    // max_seqlen (segments past a sequence's end are empty), checkpoints in the packed layout (Params::ckpt)
    const long long units = (long long)n_seq * H, total_rows = cu ? packed_rows : (long long)n_seq * T;
    if (units <= 0 || units > 0x7fffffffLL || total_rows <= 0) return GF_ERR_INVALID_ARG;
    if (total_rows >= (1LL << 31) - 64 || !ck::encode_fn()) return GF_ERR_UNSUPPORTED;
    if (!chunked_kernel_attributes()) return GF_ERR_CUDA;
    CUtensorMap tk, tv, tx, tdummy;
    const long long C = (long long)H * 64;
    if (!ck::make_map(&tk, k, total_rows, C, 64) || !ck::make_map(&tv, v, total_rows, C, 64) ||
        !ck::make_map(&tx, x, total_rows, C, 64) || !ck::make_map(&tdummy, k, total_rows, C, 16))
        return GF_ERR_CUDA;
    if (!summaries || nseg < 2) { nseg = 1; seg_chunks = (T + ck::L - 1) / ck::L; }
    ck::Params p{nullptr, k, v, x, nullptr, nullptr, state_in, nullptr, cu, T, H, summaries, seg_chunks, nseg, nullptr, c2};
    p.wait_limit_us = wait_limit_us().load(std::memory_order_relaxed);
    p.ckpt_slots = cu ? total_rows / ck::L + 2LL * n_seq : 0;
    CUtensorMap tck;                                 // the checkpoints as [slots * 64][64] bf16, 16 rows per copy
    const long long n_ckpt = cu ? (long long)H * p.ckpt_slots : units * ((T + ck::L - 1) / ck::L + 1);
    if (n_ckpt * 64 >= (1LL << 31)) return GF_ERR_UNSUPPORTED;
    if (!ck::make_map(&tck, ckpt, n_ckpt * 64, 64, 16)) return GF_ERR_CUDA;
    if (nseg > 1) {
        // few units: the segments' summaries first (every segment but the last, from a zero state), then every segment
        // side by side from its folded start state, this time keeping the states
        if (c2) ck::wkv6_chunked_kernel<true, true><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
        else ck::wkv6_chunked_kernel<true, false><<<(unsigned)(units * (nseg - 1)), ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
        launches->fetch_add(1, std::memory_order_relaxed);
        if (cudaGetLastError() != cudaSuccess) return GF_ERR_CUDA;
    }
    p.ckpt = ckpt;
    if (c2) ck::wkv6_chunked_kernel<true, true><<<(unsigned)(units * nseg), ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
    else ck::wkv6_chunked_kernel<true, false><<<(unsigned)(units * nseg), ck::THREADS, ck::SMEM_ALLOC, st>>>(tk, tk, tv, tx, tdummy, tdummy, p, tck);
    launches->fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? GF_OK : GF_ERR_CUDA;
}

// out[unit] = fold of n_fold summaries over state_in[unit] (or zero): S <- diag(D_p) S + dS_p for p = 0 .. n_fold-1,
// summaries laid out [p][unit][64 + 4096].  One CTA of 256 threads per unit; thread t owns columns of 16 rows.
__global__ void __launch_bounds__(256)
wkv6_fold_kernel(const float* __restrict__ state_in, const float* __restrict__ summaries, int n_fold, long long units,
                 float* __restrict__ out)
{
    const long long unit = blockIdx.x;
    const int j = threadIdx.x & 63, ig = threadIdx.x >> 6;             // rows 16*ig .. 16*ig+15, column j
    float S[16];
#pragma unroll
    for (int ii = 0; ii < 16; ++ii)
        S[ii] = state_in ? state_in[unit * 4096 + (size_t)(16 * ig + ii) * 64 + j] : 0.f;
    for (int pi = 0; pi < n_fold; ++pi) {
        const float* sm = summaries + ((size_t)pi * units + unit) * ck::SUMMARY_FLOATS;
#pragma unroll
        for (int ii = 0; ii < 16; ++ii)
            S[ii] = fmaf(sm[16 * ig + ii], S[ii], sm[64 + (size_t)(16 * ig + ii) * 64 + j]);
    }
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) out[unit * 4096 + (size_t)(16 * ig + ii) * 64 + j] = S[ii];
}

}  // namespace gf
