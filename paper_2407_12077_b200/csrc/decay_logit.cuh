// The decay logit of the Finch-C2 block for sm_100a: d_t = lora_omega( ddlerp_d( x_t, x_{t-1} ) ), i.e. with
//   lerp(a, b, t) = a + (b - a) t,   lora(v) = lambda + tanh(v A) B,   ddlerp(a, b) = a + (b - a) lora_d(lerp(a, b, mu_x)):
//   z_t = x_t + (x_{t-1} - x_t) mu_x                       (token shift, per channel)
//   h1  = tanh(z_t A_d)                                    [R_d]
//   m_t = x_t + (x_{t-1} - x_t) (lambda_d + h1 B_d)        (the data-dependent mix)
//   h2  = tanh(m_t A_w)                                    [R_w]
//   d_t = lambda_w + h2 B_w                                (the logit the WKV kernels take as x: w_t = exp(-exp(d_t)))
// x, d: [rows][D] bf16 with rows = B*T (x_{t-1} of a sequence's first token: x_prev[b], or zero); A_*: [D][R], B_*: [R][D]
// bf16; mu_x, lambda_*: [D] fp32.  Four skinny products (2 D (2 R_d + 2 R_w) flops per token) around elementwise
// work on a tensor that is read twice and written once: HBM-bound (4 D bytes per token when the second read of x
// hits L2), so the products run on the tensor cores and everything else is shaped to stream.
//
// One persistent CTA per SM takes an equal share of the rows (in units of 64) and walks it in tiles of 128 tokens (the last
// of 64 if the share is odd), each in three passes over the D channels, 64 at a time:
//   pass 1: z slice -> operand rows -> acc1 += z A_d[slice]                then h1 = tanh(acc1) -> operand
//   pass 2: l = h1 B_d[:, slice] -> m slice -> operand rows -> acc3 += m A_w[slice]      then h2 = tanh(acc3) -> operand
//   pass 3: d slice = lambda_w + h2 B_w[:, slice] -> bf16 -> TMA store
// Two sets of four worker warps take alternate slices, each with stages, accumulators and issuing warps of its own:
//   warp 0       TMA producer of the x rings (3 stages per set): per slice the x rows of the tile (plus the one row above
//                it) and the 64 per-channel constants of the pass; a stage is free as soon as its rows are in registers
//   warp 3       TMA producer of the weight rings (2 stages per set): free when the products that read a stage are done
//   warps 1, 2   (warp 1: tensor-memory allocation) an elected lane issues a set's z A_d, h1 B_d, h2 B_w products
//                (tcgen05.mma 128 x 64 x 16, bf16 -> fp32)
//   warps 4, 5   an elected lane issues a set's m A_w, the product that waits for the workers inside pass 2 (an issuer of
//                its own, so that the l products of later slices are not held up behind it)
//   warps 6-13   the two sets; a lane owns one token row (the accumulator row of its tensor-memory sub-partition): reads its
//                row and the row above from the swizzled x tiles, forms z / m / d for the 64 channels of the slice, 32 at a
//                time, and writes the bf16 operand row or the output slab
// z, m, h1 and h2 are A operands in tensor memory (a lane's row, two channels per column): through shared memory they were
// a third of its traffic (16 KB written and 16 KB read per slice).  A sum over slices lies in two halves, one per set.
// What bounds a slice is the chain load -> registers -> operand -> product of which two run at a time (65536 tokens x 2048
// channels: 194 us; 159 with every load left out, 160 with the stores left out).  Before (one issuer for both sets, operands
// in shared memory): 206 us; 1000 tokens 51 -> 46 us.  Twice the warps per set at half the channels each: 210 us.
// Weight tiles are the 128-byte-swizzled [64 rows][64 bf16] tiles of the prefill kernel; narrower ones (R < 64) are
// zero-filled by TMA beyond their extent.  Every wait is bounded, as in the prefill kernel.
#pragma once
#include "key_compress.cuh"
#include "wkv6_chunked.cuh"

namespace gf {
namespace dl {

using namespace ck;

constexpr int DL_NSET = 2;                             // worker sets
constexpr int DL_W0 = 6;                               // first worker warp
constexpr int DL_NWS = 4;                              // warps of a set, one per tensor-memory sub-partition
constexpr int DL_NH = 2;                               // a warp's channels of a slice come in halves of 32 (registers)
constexpr int DL_THREADS = 32 * (DL_W0 + DL_NWS * DL_NSET);
// Two rings.  The x ring holds, per slice, the tile's x rows (two swizzled 64-row tiles), the row above the tile and the
// pass's 64 per-channel constants; a worker set frees its stage as soon as the rows are in registers, so that ring
// runs a load latency ahead of the arithmetic.  The weight ring holds up to two weight tiles per slice and is freed
// by the products that read them (weights come from L2).
// Each set has rings of its own: a waiter names a phase by its parity alone, so whoever waits for a stage has to wait for
// every one of its phases (with stages that two sets use in turn, one of them asks for a phase while the other's
// before it may not have landed, and is let through).
constexpr int DL_NSX = 3, DL_NSW = 2;                  // stages per set
constexpr int DL_NACC = 2;                             // l / d accumulators in tensor memory per set: the products h1 B_d and h2 B_w
                                                       // depend on nothing the workers make, so they run this many slices ahead
constexpr int DL_XSTAGE = 2 * TILE + 1024;
constexpr int DL_OFF_PREV = 2 * TILE;                  // [64] bf16: the x row just above the tile (this slice)
constexpr int DL_OFF_VEC = 2 * TILE + 256;             // [64] fp32: mu_x / lambda_d / lambda_w of this slice
constexpr int DL_WSTAGE = 2 * TILE;
constexpr int DL_OFF_W = DL_NSET * DL_NSX * DL_XSTAGE;           // weight rings
constexpr int DL_OFF_OUT = DL_OFF_W + DL_NSET * DL_NSW * DL_WSTAGE;        // [sets][row groups][32 rows x 128 B]: output slabs of pass 3
constexpr int DL_OFF_MISC = DL_OFF_OUT + DL_NSET * 2 * TILE;     // abort word + limit, tensor-memory address, barriers
constexpr int DL_SMEM = DL_OFF_MISC + 512 + 1024;      // + slack for manual 1024-byte alignment
enum {
    DL_XFULL = 0,                      // x stage loaded
    DL_XEMPTY = DL_XFULL + DL_NSET * DL_NSX,     // ... and read into registers by the warps of its set
    DL_WFULL = DL_XEMPTY + DL_NSET * DL_NSX,     // weight stage loaded
    DL_WEMPTY = DL_WFULL + DL_NSET * DL_NSW,     // ... and the last product that reads it is done
    DL_OP_READY = DL_WEMPTY + DL_NSET * DL_NSW,  // per set: operand rows written
    DL_OP_FREE = DL_OP_READY + DL_NSET,    // per set: the product that read them is done
    DL_ACC_FULL = DL_OP_FREE + DL_NSET,    // per set and accumulator: l (pass 2) or d (pass 3) of a slice is in tensor memory
    DL_ACC_FREE = DL_ACC_FULL + DL_NSET * DL_NACC,   // ... and read back by the warps of the set
    DL_SUM_FULL = DL_ACC_FREE + DL_NSET * DL_NACC,   // both sets' partial sums of a pass complete
    DL_H_READY = DL_SUM_FULL + 1,      // h1 / h2 operand written by all worker warps
    DL_PASS2 = DL_H_READY + 1,         // per set: pass 2 of a tile has begun (its first issuer -> its second: one phase per tile)
    DL_BAR_COUNT = DL_PASS2 + DL_NSET
};
static_assert(16 + 8 * DL_BAR_COUNT <= 512, "barrier block");
static_assert(DL_SMEM <= 232448, "shared memory budget of one sm_100 CTA");
// per set: its half of the pass's sum (acc1, then acc3: every warp has read acc1 before a product of pass 2's is issued,
// and acc3 before one of the next tile's), and a ring of l (pass 2) / d (pass 3)
constexpr int DL_TM_SUM = 0, DL_TM_RING = 64 * DL_NSET;
// the A operands (lane = row, a 32-bit column = two neighbouring channels in bf16): z / m of a set, h1 / h2
constexpr int DL_TM_OP = DL_TM_RING + 64 * DL_NSET * DL_NACC, DL_TM_H = DL_TM_OP + 32 * DL_NSET;
static_assert(DL_TM_H + 32 <= 512, "tensor memory columns");
// fp32 accumulator, bf16 A (K-major) and B (MN-major), M = 128, N = 64
constexpr uint32_t DL_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((64u >> 3) << 17) | ((128u >> 4) << 24);

struct DlParams {
    long long rows;                    // B * T
    int T;                             // tokens per sequence (token shift restarts every T rows)
    int nslices;                       // D / 64
    int kd, kw;                        // 16-wide contraction steps over the two ranks: R_d / 16, R_w / 16
    const __nv_bfloat16* x_prev;       // [B][D] or NULL
    int D;
    const float *mu_x, *lambda_d, *lambda_w;
};

__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts128(uint32_t a, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// (ax + x, ay + y) rounded to a bf16 pair, the two sums in one instruction (8680 tokens x 768: 19.9 -> 19.65 us, 16982 x 1280:
// 31.4 -> 31.05)
__device__ __forceinline__ uint32_t pack_sum(float ax, float ay, uint32_t x, uint32_t y)
{
    uint32_t r;
    asm("{\n\t.reg .b64 a, b;\n\t.reg .b32 lo, hi;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\tadd.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {lo, hi}, a;\n\tcvt.rn.bf16x2.f32 %0, hi, lo;\n\t}" : "=r"(r) : "f"(ax), "f"(ay), "r"(x), "r"(y));
    return r;
}
__device__ __forceinline__ float tanh_fast(float v)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}
// D[tmem] (+)= A[tmem] * B[smem], 128 x 64 x 16, bf16 operands, fp32 accumulate: 16 contraction indices = 8 columns of A
__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// 16 / 8 consecutive 32-bit columns of this lane's row, and the wait for all such stores of the warp
__device__ __forceinline__ void tmem_st_row16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_row8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tmem_st_done() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 16 consecutive fp32 columns of this lane's accumulator row
__device__ __forceinline__ void tmem_ld_row16(uint32_t taddr, float (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr) : "memory");
}

__global__ void __launch_bounds__(DL_THREADS, 1)
decay_logit_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_x1,
                   const __grid_constant__ CUtensorMap tm_ad, const __grid_constant__ CUtensorMap tm_bd,
                   const __grid_constant__ CUtensorMap tm_aw, const __grid_constant__ CUtensorMap tm_bw,
                   const __grid_constant__ CUtensorMap tm_d32, const DlParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const uint32_t abort_flag = sbase + DL_OFF_MISC;
    auto bar = [&](int i) { return sbase + DL_OFF_MISC + 16 + 8 * i; };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // this CTA's rows, in units of 64: tiles of 128, the last of 64 if the number is odd
    const long long n_half = (p.rows + 63) / 64, r_first = n_half * blockIdx.x / gridDim.x * 64, r_end = n_half * (blockIdx.x + 1) / gridDim.x * 64;
    const int S = p.nslices;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (tid == 0) {
        for (int i = 0; i < DL_NSET * DL_NSX; ++i) {
            mbar_init(bar(DL_XFULL + i), 1);
            mbar_init(bar(DL_XEMPTY + i), DL_NWS);
        }
        for (int i = 0; i < DL_NSET * DL_NSW; ++i) {
            mbar_init(bar(DL_WFULL + i), 1);
            mbar_init(bar(DL_WEMPTY + i), 1);
        }
        for (int i = 0; i < DL_NSET; ++i) {
            mbar_init(bar(DL_OP_READY + i), DL_NWS);
            mbar_init(bar(DL_OP_FREE + i), 1);
            mbar_init(bar(DL_PASS2 + i), 1);
        }
        for (int i = 0; i < DL_NSET * DL_NACC; ++i) {
            mbar_init(bar(DL_ACC_FULL + i), 1);
            mbar_init(bar(DL_ACC_FREE + i), DL_NWS);
        }
        mbar_init(bar(DL_SUM_FULL), DL_NSET);
        mbar_init(bar(DL_H_READY), DL_NWS * DL_NSET);
        sts32(abort_flag, 0u);
        sts32(abort_flag + 4, WAIT_LIMIT_US);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 1) tmem_alloc(sbase + DL_OFF_MISC + 8, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = lds32(sbase + DL_OFF_MISC + 8);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ring positions: the set's n-th slice over all passes and tiles
    auto xslot = [&](int set, int n) { return set * DL_NSX + n % DL_NSX; };
    auto wslot = [&](int set, int n) { return set * DL_NSW + n % DL_NSW; };
    auto wstage = [&](int slot) { return sbase + DL_OFF_W + slot * DL_WSTAGE; };

    if (warp == 0) {
        // ============================== TMA producer: x rows and per-channel constants ==============================
        int n[DL_NSET] = {};                                 // slices issued so far, per set
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128) {
            const int row0 = (int)r;
            const bool whole = r_end - r > 64;
            for (int pass = 0; pass < 3 && alive; ++pass)
                for (int s = 0; s < S; ++s) {
                    const int set = s % DL_NSET, c = set ? n[1] : n[0], slot = xslot(set, c);
                    if (c >= DL_NSX && !mbar_wait_warp(bar(DL_XEMPTY + slot), ((c / DL_NSX) + 1) & 1, abort_flag)) { alive = false; break; }
                    const uint32_t dst = sbase + slot * DL_XSTAGE, full = bar(DL_XFULL + slot);
                    if (elect_one()) {
                        const float* vec = pass == 0 ? p.mu_x : pass == 1 ? p.lambda_d : p.lambda_w;
                        if (pass < 2) {
                            mbar_expect_tx(full, (whole ? 2 * TILE : TILE) + 128 + 256);
                            tma_load_2d(dst, &tm_x, 64 * s, row0, full);
                            if (whole) tma_load_2d(dst + TILE, &tm_x, 64 * s, row0 + 64, full);
                            tma_load_2d(dst + DL_OFF_PREV, &tm_x1, 64 * s, row0 - 1, full);      // (row -1 reads as zero)
                        } else {
                            mbar_expect_tx(full, 256);
                        }
                        bulk_load_1d(dst + DL_OFF_VEC, vec + 64 * s, 256, full);
                    }
                    __syncwarp();
                    if (set) ++n[1]; else ++n[0];
                }
        }
        // do not leave while copies into this CTA's shared memory may still be in flight
        for (int set = 0; set < DL_NSET; ++set)
            for (int c = max(0, n[set] - DL_NSX); c < n[set]; ++c)
                mbar_wait_warp(bar(DL_XFULL + xslot(set, c)), (c / DL_NSX) & 1, abort_flag, false);
    } else if (warp == 3) {
        // ============================== TMA producer: weight tiles ==============================
        int n[DL_NSET] = {};
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128)
            for (int pass = 0; pass < 3 && alive; ++pass)
                for (int s = 0; s < S; ++s) {
                    const int set = s % DL_NSET, c = set ? n[1] : n[0], slot = wslot(set, c);
                    if (c >= DL_NSW && !mbar_wait_warp(bar(DL_WEMPTY + slot), ((c / DL_NSW) + 1) & 1, abort_flag)) { alive = false; break; }
                    const uint32_t dst = wstage(slot), full = bar(DL_WFULL + slot);
                    if (elect_one()) {
                        if (pass == 0) {
                            mbar_expect_tx(full, TILE);
                            tma_load_2d(dst, &tm_ad, 0, 64 * s, full);
                        } else if (pass == 1) {
                            mbar_expect_tx(full, 2 * TILE);
                            tma_load_2d(dst, &tm_bd, 64 * s, 0, full);
                            tma_load_2d(dst + TILE, &tm_aw, 0, 64 * s, full);
                        } else {
                            mbar_expect_tx(full, TILE);
                            tma_load_2d(dst, &tm_bw, 64 * s, 0, full);
                        }
                    }
                    __syncwarp();
                    if (set) ++n[1]; else ++n[0];
                }
        for (int set = 0; set < DL_NSET; ++set)
            for (int c = max(0, n[set] - DL_NSW); c < n[set]; ++c)
                mbar_wait_warp(bar(DL_WFULL + wslot(set, c)), (c / DL_NSW) & 1, abort_flag, false);
    } else if (warp == 1 || warp == 2) {
        // ============================== MMA issuers: z A_d, h1 B_d, h2 B_w of one set's slices ==============================
        const int set = warp - 1;
        const int n_own = (S - set + DL_NSET - 1) / DL_NSET;         // slices of this set (set, set + 2, ...)
        const uint32_t tsum = tmem + DL_TM_SUM + 64 * set, tring = tmem + DL_TM_RING + 64 * DL_NACC * set;
        int n = 0;                                           // ring position
        int op_uses = 0;                                     // operand tiles of this set consumed
        int an = 0;                                          // l / d accumulators of this set produced so far
        bool alive = true;
        auto weights_in = [&](int c) { return mbar_wait_warp(bar(DL_WFULL + wslot(set, c)), (c / DL_NSW) & 1, abort_flag); };
        auto acc_free = [&](int n) { return n < DL_NACC || mbar_wait_warp(bar(DL_ACC_FREE + DL_NACC * set + n % DL_NACC), ((n / DL_NACC) + 1) & 1, abort_flag); };
        const uint32_t th = tmem + DL_TM_H, ta = tmem + DL_TM_OP + 32 * set;
        for (long long r = r_first; r < r_end && alive; r += 128) {
            // ---- pass 1: acc1 += z A_d[slice]
            for (int s = set; s < S; s += DL_NSET, ++n) {
                const int i = wslot(set, n);
                if (!weights_in(n) || !mbar_wait_warp(bar(DL_OP_READY + set), op_uses & 1, abort_flag)) { alive = false; break; }
                ++op_uses;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t db = smem_desc(wstage(i));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma_ta(tsum, ta + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, (s > set || kk > 0) ? 1u : 0u);
                    tc_commit(bar(DL_OP_FREE + set));
                    tc_commit(bar(DL_WEMPTY + i));
                    if (s + DL_NSET >= S) tc_commit(bar(DL_SUM_FULL));
                }
                __syncwarp();
            }
            if (!alive) break;
            if (n_own == 0 && elect_one()) mbar_arrive(bar(DL_SUM_FULL));        // (one slice: the other set's sum is all)
            __syncwarp();
            // ---- pass 2: l = h1 B_d[:, slice] (the set's other issuer follows with acc3 += m A_w[slice] and frees the stage)
            if (!mbar_wait_warp(bar(DL_H_READY), 0, abort_flag)) break;          // (two uses per tile: parities 0, 1)
            tc_fence_after();
            if (elect_one()) mbar_arrive(bar(DL_PASS2 + set));                    // every operand-row phase of pass 1 is over
            __syncwarp();
            for (int s = set; s < S; s += DL_NSET, ++an, ++n) {
                const int i = wslot(set, n), a = an % DL_NACC;
                if (!weights_in(n) || !acc_free(an)) { alive = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t db = smem_desc(wstage(i));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        if (kk < p.kd) tc_mma_ta(tring + 64 * a, th + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, kk > 0 ? 1u : 0u);
                    tc_commit(bar(DL_ACC_FULL + DL_NACC * set + a));
                }
                __syncwarp();
            }
            op_uses += n_own;                                 // (the set's other issuer consumes these slices' operand rows)
            if (!alive) break;
            // ---- pass 3: d slice = h2 B_w[:, slice]
            if (!mbar_wait_warp(bar(DL_H_READY), 1, abort_flag)) break;
            tc_fence_after();
            for (int s = set; s < S; s += DL_NSET, ++an, ++n) {
                const int i = wslot(set, n), a = an % DL_NACC;
                if (!weights_in(n) || !acc_free(an)) { alive = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t db = smem_desc(wstage(i));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        if (kk < p.kw) tc_mma_ta(tring + 64 * a, th + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, kk > 0 ? 1u : 0u);
                    tc_commit(bar(DL_ACC_FULL + DL_NACC * set + a));
                    tc_commit(bar(DL_WEMPTY + i));
                }
                __syncwarp();
            }
        }
    } else if (warp == 4 || warp == 5) {
        // ============================== MMA issuers: m A_w (pass 2) of one set's slices ==============================
        const int set = warp - 4;
        const int n_own = (S - set + DL_NSET - 1) / DL_NSET;
        const uint32_t tsum = tmem + DL_TM_SUM + 64 * set;
        const uint32_t ta = tmem + DL_TM_OP + 32 * set;
        int ti = 0, op_uses = 0;
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128, ++ti) {
            // A wait names a phase by its parity alone, so it must not start more than one phase ahead of the barrier:
            // the operand-row barriers go through pass 1's phases first (the other issuer's), hence the go-ahead.
            if (!mbar_wait_warp(bar(DL_PASS2 + set), ti & 1, abort_flag)) break;
            op_uses += n_own;                                            // pass 1's uses of the operand rows
            int n = (ti * 3 + 1) * n_own;                                 // ring position of pass 2, first slice
            for (int s = set; s < S; s += DL_NSET, ++n) {
                const int i = wslot(set, n);
                if (!mbar_wait_warp(bar(DL_OP_READY + set), op_uses & 1, abort_flag)) { alive = false; break; }
                ++op_uses;
                // (its weights are there: the other issuer saw this phase complete before it made the l this operand was built
                // from, and the next one waits for this product)
                if (!mbar_wait_warp(bar(DL_WFULL + i), (n / DL_NSW) & 1, abort_flag)) { alive = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t db = smem_desc(wstage(i) + TILE);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma_ta(tsum, ta + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, (s > set || kk > 0) ? 1u : 0u);
                    tc_commit(bar(DL_OP_FREE + set));
                    tc_commit(bar(DL_WEMPTY + i));
                    if (s + DL_NSET >= S) tc_commit(bar(DL_SUM_FULL));
                }
                __syncwarp();
            }
            if (n_own == 0 && elect_one()) mbar_arrive(bar(DL_SUM_FULL));
            __syncwarp();
        }
    } else {
        // ============================== worker warps ==============================
        const int set = (warp - DL_W0) / DL_NWS;         // takes the slices s with s mod DL_NSET == set
        const int n_own = (S - set + DL_NSET - 1) / DL_NSET;
        const uint32_t tring = tmem + DL_TM_RING + 64 * DL_NACC * set;
        const int sp = warp & 3;                         // tensor-memory sub-partition: accumulator rows 32*sp .. 32*sp+31
        const int row = 32 * sp + lane;                  // this lane's token row inside the tile
        const uint32_t tlane = (uint32_t)(32 * sp) << 16;
        const uint32_t own_tile = (uint32_t)(row >> 6) * TILE, own_row = (uint32_t)(row & 63);
        const uint32_t up_tile = (uint32_t)((row - 1) >> 6) * TILE, up_row = (uint32_t)((row - 1) & 63);   // (row > 0)
        const uint32_t own_xor = (own_row & 7) << 4;
        const uint32_t slab0 = sbase + DL_OFF_OUT + set * 2 * TILE + sp * 4096;     // pass 3: this warp's output slab, 32 rows x 128 B
        int op_uses = 0;
        bool alive = true;

        // h = tanh(acc), acc the sum of the sets' halves, for this warp's 32 rows and its share of the 64 columns -> bf16
        // operand rows
        auto squash = [&]() {
#pragma unroll
            for (int g = 0; g < DL_NH; ++g) {
                const int c0 = 32 * set + 16 * g;
                float a[16], b[16];
                tmem_ld_row16(tmem + tlane + DL_TM_SUM + c0, a);
                if (S > 1) tmem_ld_row16(tmem + tlane + DL_TM_SUM + 64 + c0, b);
#pragma unroll
                for (int e = 0; e < 16; ++e) a[e] = S > 1 ? a[e] + b[e] : a[e];
                uint32_t ow[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) ow[e] = pack_bf16(tanh_fast(a[2 * e]), tanh_fast(a[2 * e + 1]));
                tmem_st_row8(tmem + tlane + DL_TM_H + c0 / 2, ow);
            }
            tmem_st_done();
        };
        static_assert(DL_NSET == 2, "the sum of two halves");

        int it = 0, ti = 0;
        for (long long r = r_first; r < r_end && alive; r += 128, ++ti) {
            const long long tok = r + row;
            const bool live = r + 32 * sp < r_end;       // (a tile of 64 rows: two row groups only keep the barriers company)
            const bool seq_start = (tok % p.T) == 0;     // the row above belongs to another sequence: x_prev or zero
            const bool any_start = __any_sync(0xffffffffu, seq_start);
            const __nv_bfloat16* gp0 = (seq_start && p.x_prev && tok < p.rows) ? p.x_prev + (tok / p.T) * (long long)p.D : nullptr;
            // ---- passes 1 and 2: out = x + (x_above - x) * mix, mix = the pass's constants (+ l from tensor memory in pass 2).
            // The interpolation runs on packed bf16 pairs (difference, then one fused multiply-add with a single rounding):
            // its inputs and its output are bf16 anyway, and the mix is smooth in them.
            for (int pass = 0; pass < 2 && alive; ++pass) {
                for (int s = set; s < S; s += DL_NSET, ++it) {
                    const int i = xslot(set, it);
                    const uint32_t stage = sbase + i * DL_XSTAGE;
                    if (!mbar_wait(bar(DL_XFULL + i), (it / DL_NSX) & 1, abort_flag)) { alive = false; break; }
                    const int an = ti * 2 * n_own + s / DL_NSET, acc = an % DL_NACC;             // this slice's l: the set's an-th accumulator
                    if (pass == 1) {
                        if (!mbar_wait(bar(DL_ACC_FULL + DL_NACC * set + acc), (an / DL_NACC) & 1, abort_flag)) { alive = false; break; }
                        tc_fence_after();
                    }
                    // this lane's row and the row above it (inside the tiles, or the extra row of the stage for the tile's
                    // first row)
                    const uint32_t up_base = row == 0 ? stage + DL_OFF_PREV : stage + up_tile + up_row * 128;
                    const uint32_t up_xor = row == 0 ? 0u : (up_row & 7) << 4;
                    const uint32_t own_base = stage + own_tile + own_row * 128;
                    if (!live) {
                        if (pass == 1) { tc_fence_before(); __syncwarp(); mbar_arrive_if(bar(DL_ACC_FREE + DL_NACC * set + acc), lane == 0); }
                        __syncwarp();
                        mbar_arrive_if(bar(DL_XEMPTY + i), lane == 0);
                        if (op_uses >= 1 && !mbar_wait(bar(DL_OP_FREE + set), (op_uses - 1) & 1, abort_flag)) { alive = false; break; }
                    } else
#pragma unroll
                    for (int g = 0; g < DL_NH; ++g) {
                        const int hf = g;
                        uint32_t mixw[16];               // the mix of 32 channels as bf16 pairs
                        if (pass == 1) {
                            uint32_t l[32];
                            kc::tmem_ld_row32(tring + tlane + 64 * acc + 32 * hf, l);
                            if (g == DL_NH - 1) {        // the accumulator row has been read: hand it back
                                tc_fence_before();
                                __syncwarp();
                                mbar_arrive_if(bar(DL_ACC_FREE + DL_NACC * set + acc), lane == 0);
                            }
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 v4 = ldsf4(stage + DL_OFF_VEC + 128 * hf + 16 * q);
                                mixw[2 * q] = pack_sum(v4.x, v4.y, l[4 * q], l[4 * q + 1]);
                                mixw[2 * q + 1] = pack_sum(v4.z, v4.w, l[4 * q + 2], l[4 * q + 3]);
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 v4 = ldsf4(stage + DL_OFF_VEC + 128 * hf + 16 * q);
                                mixw[2 * q] = pack_bf16(v4.x, v4.y);
                                mixw[2 * q + 1] = pack_bf16(v4.z, v4.w);
                            }
                        }
                        uint4 a[4], b[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t o = (uint32_t)((4 * hf + q) << 4);
                            a[q] = lds128(own_base + (o ^ own_xor));
                            b[q] = lds128(up_base + (o ^ up_xor));
                        }
                        if (g == DL_NH - 1) {            // all in registers: the stage is free for a later slice
                            __syncwarp();
                            mbar_arrive_if(bar(DL_XEMPTY + i), lane == 0);
                        }
                        if (any_start && seq_start) {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                b[q] = gp0 ? *reinterpret_cast<const uint4*>(gp0 + 64 * s + 32 * hf + 8 * q) : make_uint4(0u, 0u, 0u, 0u);
                        }
                        // the operand rows: free of the product that read them last
                        if (g == 0 && op_uses >= 1 && !mbar_wait(bar(DL_OP_FREE + set), (op_uses - 1) & 1, abort_flag)) { alive = false; break; }
                        uint32_t ow[16];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t aw[4] = {a[q].x, a[q].y, a[q].z, a[q].w}, bw[4] = {b[q].x, b[q].y, b[q].z, b[q].w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                uint32_t delta;
                                asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(delta) : "r"(bw[e]), "r"(aw[e]));
                                asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(ow[4 * q + e]) : "r"(delta), "r"(mixw[4 * q + e]), "r"(aw[e]));
                            }
                        }
                        if (g == 0) tc_fence_after();
                        __syncwarp();
                        tmem_st_row16(tmem + tlane + DL_TM_OP + 32 * set + 16 * hf, ow);
                    }
                    if (!alive) break;
                    ++op_uses;
                    tmem_st_done();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bar(DL_OP_READY + set), lane == 0);
                }
                if (!alive) break;
                // the pass's low-rank sum is complete: squash it into the operand of the next product
                if (!mbar_wait(bar(DL_SUM_FULL), pass, abort_flag)) { alive = false; break; }      // (two uses per tile)
                tc_fence_after();
                if (live) squash();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_if(bar(DL_H_READY), lane == 0);
            }
            if (!alive) break;
            // ---- pass 3: d slice -> bf16 slab -> TMA store
            for (int s = set; s < S; s += DL_NSET, ++it) {
                const int i = xslot(set, it);
                const uint32_t stage = sbase + i * DL_XSTAGE;
                if (!mbar_wait(bar(DL_XFULL + i), (it / DL_NSX) & 1, abort_flag)) { alive = false; break; }
                const int an = ti * 2 * n_own + n_own + s / DL_NSET, acc = an % DL_NACC;         // this slice's d
                if (!mbar_wait(bar(DL_ACC_FULL + DL_NACC * set + acc), (an / DL_NACC) & 1, abort_flag)) { alive = false; break; }
                tc_fence_after();
                if (!live) {
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bar(DL_ACC_FREE + DL_NACC * set + acc), lane == 0);
                    mbar_arrive_if(bar(DL_XEMPTY + i), lane == 0);
                    continue;
                }
                if (lane == 0) bulk_wait_read<0>();      // this warp's previous stores have finished reading the slabs
                __syncwarp();
#pragma unroll
                for (int g = 0; g < DL_NH; ++g) {
                    const int hf = g;
                    uint32_t v[32];
                    kc::tmem_ld_row32(tring + tlane + 64 * acc + 32 * hf, v);
                    if (g == DL_NH - 1) {
                        tc_fence_before();
                        __syncwarp();
                        mbar_arrive_if(bar(DL_ACC_FREE + DL_NACC * set + acc), lane == 0);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 la = ldsf4(stage + DL_OFF_VEC + 128 * hf + 32 * q), lb = ldsf4(stage + DL_OFF_VEC + 128 * hf + 32 * q + 16);
                        sts128(slab0 + swz(lane, (4 * hf + q) << 4),
                               make_uint4(pack_sum(la.x, la.y, v[8 * q], v[8 * q + 1]), pack_sum(la.z, la.w, v[8 * q + 2], v[8 * q + 3]),
                                          pack_sum(lb.x, lb.y, v[8 * q + 4], v[8 * q + 5]), pack_sum(lb.z, lb.w, v[8 * q + 6], v[8 * q + 7])));
                    }
                }
                __syncwarp();
                mbar_arrive_if(bar(DL_XEMPTY + i), lane == 0);
                fence_proxy_async();
                __syncwarp();
                const long long grow = r + 32 * sp;
                if (lane == 0 && grow < p.rows) {
                    tma_store_2d(&tm_d32, 64 * s, (int)grow, slab0);
                    bulk_commit();
                }
            }
            if (!alive) break;
        }
        if (lane == 0) bulk_wait<0>();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// [rows][cols] bf16 tensor map with a box of box_rows x box_cols (box_cols * 2 bytes <= 128)
inline bool make_map_box(CUtensorMap* tm, const void* base, long long rows, long long cols, int box_rows, int box_cols, CUtensorMapSwizzle swizzle)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dl

// d = lora_omega(ddlerp_d(x, shifted x)) over rows = B*T tokens of D channels; see the top of this file.
inline gf_status_t decay_logit(const __nv_bfloat16* x, const __nv_bfloat16* x_prev, const float* mu_x,
                               const __nv_bfloat16* A_d, const __nv_bfloat16* B_d, const float* lambda_d,
                               const __nv_bfloat16* A_w, const __nv_bfloat16* B_w, const float* lambda_w,
                               __nv_bfloat16* d, int B, int T, int D, int Rd, int Rw, cudaStream_t st,
                               std::atomic<uint64_t>* launches)
{
    const long long rows = (long long)B * T;
    static PerDeviceFlag attr_set;
    const int dev = current_device();
    if (dev < 0) return GF_ERR_CUDA;
    if (!attr_set.is_set(dev)) {
        if (cudaFuncSetAttribute(dl::decay_logit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dl::DL_SMEM) != cudaSuccess)
            return GF_ERR_CUDA;
        attr_set.set(dev);
    }
    CUtensorMap tx, tx1, tad, tbd, taw, tbw, td;
    constexpr CUtensorMapSwizzle sw128 = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!dl::make_map_box(&tx, x, rows, D, 64, 64, sw128) || !dl::make_map_box(&tx1, x, rows, D, 1, 64, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !dl::make_map_box(&tad, A_d, D, Rd, 64, 64, sw128) || !dl::make_map_box(&tbd, B_d, Rd, D, 64, 64, sw128) ||
        !dl::make_map_box(&taw, A_w, D, Rw, 64, 64, sw128) || !dl::make_map_box(&tbw, B_w, Rw, D, 64, 64, sw128) ||
        !dl::make_map_box(&td, d, rows, D, 32, 64, sw128))
        return GF_ERR_CUDA;
    dl::DlParams p{rows, T, D / 64, Rd / 16, Rw / 16, x_prev, D, mu_x, lambda_d, lambda_w};
    const long long n_half = (rows + 63) / 64;
    const int n_sm = sm_count();
    const unsigned grid = (unsigned)(n_half < n_sm ? n_half : n_sm);
    const cudaError_t e = launch_pdl(dl::decay_logit_kernel, grid, dl::DL_THREADS, dl::DL_SMEM, st, tx, tx1, tad, tbd, taw, tbw, td, p);
    launches->fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? GF_OK : GF_ERR_CUDA;
}

}  // namespace gf
