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
// Four sets of four worker warps take the slices in turn, each with a tensor-memory operand of its own:
//   warp 0       TMA producer of the x ring (8 stages, two per set): per slice the x rows of the tile (plus the one row above
//                it) and the 64 per-channel constants of the pass; a stage is free as soon as its rows are in registers (pass 3: its
//                room takes the output rows, and it is free when the store has read them)
//   warps 1, 20  TMA producers of the weight rings (A_d, A_w: 5 stages; B_d, B_w: 3 per issuer): free when the product that reads a stage is done
//   warp 2       an elected lane issues the products that wait for the workers, z A_d and m A_w (tcgen05.mma 128 x 64 x 16,
//                bf16 -> fp32; tensor-memory allocation)
//   warps 3, 21  an elected lane issues h1 B_d and h2 B_w of the even, the odd slices
//   warps 4-19   the four sets; a lane owns one token row (the accumulator row of its tensor-memory sub-partition): reads its
//                row and the row above from the swizzled x tiles, forms z / m / d for the 64 channels of the slice, 32 at a
//                time (mix first, so that an accumulator is soon free), and writes the bf16 operand row or the output slab
// z, m, h1 and h2 are A operands in tensor memory (a lane's row, two channels per column): through shared memory they were
// a third of its traffic (16 KB written and 16 KB read per slice).
// What bounds a slice is the chain load -> registers -> operand -> product, through warps that each spend 300-400 cycles per slice on
// their part: 870 cycles a slice and pass with every set in flight, and 780 with one tile on an idle SM.  us per call, two sets of four warps on
// rings of two weight stages each -> four sets -> a weight ring per issuer -> a producer and an issuer more:
//   65536 tokens x 2048 channels 191 -> 196 -> 179 -> 175;  1000 x 2048 46.4 -> 43.5 -> 41.4 -> 40.0;  32 x 271 x 2048 50.5 -> 46.3 -> 45.7 -> 43.6;
//   8680 x 768 20.1 -> 20.5 -> 19.6 -> 19.3.
// That form had one chain of sums for all slices and an accumulator per set.  With the sums of the even and the odd slices apart, as two
// sets had them, three accumulators are what tensor memory has room for.  us per call in a graph, two sets -> one chain -> present form:
//   65536 x 2048 189.7 -> 173.9 -> 173.0;  19500 x 2048 90.1 -> 82.0 -> 83.2;  9400 x 2048 41.5 -> 36.3 -> 37.9;
//   65536 x 1280 120.6 -> 116.0 -> 115.7;  18000 x 1280 30.2 -> 30.7 -> 30.2;  40 x 1280 26.9 -> 23.6 -> 25.2;
//   65536 x 768 78.7 -> 78.6 -> 79.2;  18000 x 768 20.0 -> 20.7 -> 20.3;  40 x 768 17.8 -> 16.2 -> 17.4;  18000 x 256 10.7 -> 12.1 -> 12.3.
// (l read in quarters of a slice, so that an accumulator is held for most of it: 40 x 768 17.8, 65536 x 2048 177; read as a whole first
// 17.5 and 173.7, with two accumulators 17.6 and 175; slices 2 and 3 of a pass in the idle halves of the sum 17.8 and 178.)
// (With one ring for both kinds of weights a slice's B_d, which its l needs early, waited for the slot of an A_w whose product comes a worker's
// time later.)  Not better: the sum of pass 1 in an accumulator per set (175.6), rings of 5 + 6 stages with one producer (181), asking for the
// operand rows after more of the slice (174 to 205: registers), an extra commit saved per slice at rings of 4 (192).  The three passes
// as a pipeline over tiles, with pass 1 a product of raw rows with scaled weights, ran at 215: rings of two stages are all that fits then.
// Weight tiles are the 128-byte-swizzled [64 rows][64 bf16] tiles of the prefill kernel; narrower ones (R < 64) are
// zero-filled by TMA beyond their extent.  Every wait is bounded, as in the prefill kernel.
#pragma once
#include "key_compress.cuh"
#include "wkv6_chunked.cuh"

namespace gf {
namespace dl {

using namespace ck;

constexpr int DL_NSET = 4;                             // worker sets
constexpr int DL_W0 = 4;                               // first worker warp
constexpr int DL_NWS = 4;                              // warps of a set, one per tensor-memory sub-partition
constexpr int DL_WB = DL_W0 + DL_NWS * DL_NSET;        // last warp: the producer of the B weights
constexpr int DL_THREADS = 32 * (DL_WB + 2);
// Slices are counted through all passes and tiles; slice n belongs to set n mod 4 and takes stage n mod 8 of the x ring, so a stage
// always serves the same set.  (A wait names a phase by its parity alone, so whoever waits on a barrier has to wait for every one of its phases.)
constexpr int DL_NSX = 8, DL_NSA = 5, DL_NSB = 3;
static_assert(DL_NSX % DL_NSET == 0, "a stage serves one set");
constexpr int DL_XSTAGE = 2 * TILE + 1024;
constexpr int DL_OFF_PREV = 2 * TILE;                  // [64] bf16: the x row just above the tile (this slice)
constexpr int DL_OFF_VEC = 2 * TILE + 256;             // [64] fp32: mu_x / lambda_d / lambda_w of this slice
constexpr int DL_OFF_A = DL_NSX * DL_XSTAGE;           // weight rings: A_d, A_w slices; B_d, B_w slices
constexpr int DL_OFF_B = DL_OFF_A + DL_NSA * TILE;
constexpr int DL_OFF_MISC = DL_OFF_B + 2 * DL_NSB * TILE;       // abort word + limit, tensor-memory address, barriers
constexpr int DL_SMEM = DL_OFF_MISC + 512 + 1024;      // + slack for manual 1024-byte alignment
enum {
    DL_XFULL = 0,                      // x stage loaded
    DL_XEMPTY = DL_XFULL + DL_NSX,     // ... and read into registers by the warps of its set
    DL_AFULL = DL_XEMPTY + DL_NSX,     // A weight stage loaded
    DL_AEMPTY = DL_AFULL + DL_NSA,     // ... and the product that reads it is done
    DL_BFULL = DL_AEMPTY + DL_NSA,     // B weights
    DL_BEMPTY = DL_BFULL + 2 * DL_NSB,
    DL_OP_READY = DL_BEMPTY + 2 * DL_NSB,  // per set: operand rows written
    DL_OP_FREE = DL_OP_READY + DL_NSET,    // per set: the product that read them is done
    DL_ACC_FULL = DL_OP_FREE + DL_NSET,    // per set: l (pass 2) or d (pass 3) of a slice is in tensor memory
    DL_ACC_FREE = DL_ACC_FULL + DL_NSET,   // ... and read back by the warps of the set
    DL_TURN = DL_ACC_FREE + DL_NSET,       // per issuer of h B: the accumulator of its slice was free
    DL_SUM_FULL = DL_TURN + 2,             // the sum of a pass complete
    DL_H1_READY = DL_SUM_FULL + 1,     // h1 operand written by all worker warps: one phase per tile
    DL_H2_READY = DL_H1_READY + 1,     // h2 operand: the same (and every warp has read acc3)
    DL_H_FREE = DL_H2_READY + 1,       // the last product of a tile that reads h2 is done
    DL_BAR_COUNT = DL_H_FREE + 1
};
static_assert(16 + 8 * DL_BAR_COUNT <= 512, "barrier block");
static_assert(DL_SMEM <= 232448, "shared memory budget of one sm_100 CTA");
// the sum of a pass in two halves, its even and its odd slices, which keeps the chains of additions short (acc1, then acc3: every
// warp has read acc1 before a product of pass 2's is issued, and acc3 before one of the next tile's: DL_H1_READY, DL_H2_READY); a
// ring of accumulators for l (pass 2) / d (pass 3) in the order of the slices; the A operands (lane = row, a 32-bit column = two
// neighbouring channels in bf16): z / m of a set, h1 / h2
constexpr int DL_NACC = 3;
constexpr int DL_TM_SUM = 0, DL_TM_ACC = 2 * 64, DL_TM_OP = DL_TM_ACC + 64 * DL_NACC, DL_TM_H = DL_TM_OP + 32 * DL_NSET;
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
        for (int i = 0; i < DL_NSX; ++i) {
            mbar_init(bar(DL_XFULL + i), 1);
            mbar_init(bar(DL_XEMPTY + i), DL_NWS);
        }
        for (int i = 0; i < 2 * DL_NSA; ++i) mbar_init(bar(DL_AFULL + i), 1);
        for (int i = 0; i < 4 * DL_NSB; ++i) mbar_init(bar(DL_BFULL + i), 1);
        for (int i = 0; i < DL_NSET; ++i) {
            mbar_init(bar(DL_OP_READY + i), DL_NWS);
            mbar_init(bar(DL_OP_FREE + i), 1);
            mbar_init(bar(DL_ACC_FULL + i), 1);
        }
        for (int i = 0; i < DL_NSET; ++i) mbar_init(bar(DL_ACC_FREE + i), DL_NWS);
        mbar_init(bar(DL_TURN), 1);
        mbar_init(bar(DL_TURN + 1), 1);
        mbar_init(bar(DL_SUM_FULL), 1);
        mbar_init(bar(DL_H1_READY), DL_NWS * DL_NSET);
        mbar_init(bar(DL_H2_READY), DL_NWS * DL_NSET);
        mbar_init(bar(DL_H_FREE), 2);
        sts32(abort_flag, 0u);
        sts32(abort_flag + 4, WAIT_LIMIT_US);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 2) tmem_alloc(sbase + DL_OFF_MISC + 8, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = lds32(sbase + DL_OFF_MISC + 8);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    auto wait = [&](int b, int phase) { return mbar_wait(bar(b), phase & 1, abort_flag); };
    auto wait_warp = [&](int b, int phase) { return mbar_wait_warp(bar(b), phase & 1, abort_flag); };
    auto xstage = [&](int n) { return sbase + (n & (DL_NSX - 1)) * DL_XSTAGE; };
    auto astage = [&](int i) { return sbase + DL_OFF_A + i * TILE; };
    auto bstage = [&](int i) { return sbase + DL_OFF_B + i * TILE; };

    if (warp == 0) {
        // ============================== TMA producer: x rows and per-channel constants ==============================
        int n = 0;
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128) {
            const int row0 = (int)r;
            const bool whole = r_end - r > 64;
            for (int pass = 0; pass < 3 && alive; ++pass)
                for (int s = 0; s < S; ++s, ++n) {
                    if (n >= DL_NSX && !wait_warp(DL_XEMPTY + (n & (DL_NSX - 1)), n / DL_NSX - 1)) { alive = false; break; }
                    const uint32_t dst = xstage(n), full = bar(DL_XFULL + (n & (DL_NSX - 1)));
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
                }
        }
        // do not leave while copies into this CTA's shared memory may still be in flight
        for (int c = max(0, n - DL_NSX); c < n; ++c) mbar_wait_warp(bar(DL_XFULL + (c & (DL_NSX - 1))), (c / DL_NSX) & 1, abort_flag, false);
    } else if (warp == 1) {
        // ============================== TMA producer: A_d, A_w tiles ==============================
        int n = 0, ia = 0, pa = 1;                           // tiles issued; ring position and the parity of its last release
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128)
            for (int pass = 0; pass < 2 && alive; ++pass)
                for (int s = 0; s < S; ++s, ++n) {
                    if (n >= DL_NSA && !wait_warp(DL_AEMPTY + ia, pa)) { alive = false; break; }
                    if (elect_one()) {
                        const uint32_t full = bar(DL_AFULL + ia);
                        mbar_expect_tx(full, TILE);
                        tma_load_2d(astage(ia), pass == 0 ? &tm_ad : &tm_aw, 0, 64 * s, full);
                    }
                    __syncwarp();
                    if (++ia == DL_NSA) { ia = 0; pa ^= 1; }
                }
        for (int c = max(0, n - DL_NSA); c < n; ++c) mbar_wait_warp(bar(DL_AFULL + c % DL_NSA), (c / DL_NSA) & 1, abort_flag, false);
    } else if (warp == DL_WB) {
        // ============================== TMA producer: B_d, B_w tiles ==============================
        int n = 0, i0 = 0, i1 = 0, m0 = 0, m1 = 0;           // per issuer: tiles issued, ring position
        bool alive = true;
        auto phase = [](int m) { return m / DL_NSB; };
        for (long long r = r_first; r < r_end && alive; r += 128) {
            n += S;
            for (int pass = 1; pass < 3 && alive; ++pass)
                for (int s = 0; s < S; ++s, ++n) {
                    const bool odd = n & 1;
                    const int m = odd ? m1 : m0, slot = odd ? DL_NSB + i1 : i0;
                    if (m >= DL_NSB && !wait_warp(DL_BEMPTY + slot, phase(m) - 1)) { alive = false; break; }
                    if (elect_one()) {
                        const uint32_t full = bar(DL_BFULL + slot);
                        mbar_expect_tx(full, TILE);
                        tma_load_2d(bstage(slot), pass == 1 ? &tm_bd : &tm_bw, 64 * s, 0, full);
                    }
                    __syncwarp();
                    if (odd) { ++m1; if (++i1 == DL_NSB) i1 = 0; }
                    else { ++m0; if (++i0 == DL_NSB) i0 = 0; }
                }
        }
        for (int c = max(0, m0 - DL_NSB); c < m0; ++c) mbar_wait_warp(bar(DL_BFULL + c % DL_NSB), phase(c) & 1, abort_flag, false);
        for (int c = max(0, m1 - DL_NSB); c < m1; ++c) mbar_wait_warp(bar(DL_BFULL + DL_NSB + c % DL_NSB), phase(c) & 1, abort_flag, false);
    } else if (warp == 2) {
        // ============================== MMA issuer: sum += z A_d (pass 1), sum += m A_w (pass 2) ==============================
        int n = 0, ia = 0, pa = 0;                           // (A ring position and its phase)
        uint32_t phases = 0;                                 // bit: parity of the set's next operand
        bool alive = true;
        int ti = 0;
        for (long long r = r_first; r < r_end && alive; r += 128, ++ti) {
            // Every warp has read the sum of the tile before.  (Where a set has no slice in pass 3, its next operand does not say so.)
            if (ti > 0 && !wait_warp(DL_H2_READY, ti - 1)) break;
            for (int pass = 0; pass < 2 && alive; ++pass)
                for (int s = 0; s < S; ++s, ++n) {
                    const int set = n & (DL_NSET - 1);
                    if (!wait_warp(DL_OP_READY + set, phases >> set)) { alive = false; break; }
                    phases ^= 1u << set;
                    if (!wait_warp(DL_AFULL + ia, pa)) { alive = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t db = smem_desc(astage(ia));
                        const uint32_t ta = tmem + DL_TM_OP + 32 * set;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            tc_mma_ta(tmem + DL_TM_SUM + 64 * (s & 1), ta + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, (s > 1 || kk > 0) ? 1u : 0u);
                        tc_commit(bar(DL_OP_FREE + set));
                        tc_commit(bar(DL_AEMPTY + ia));
                        if (s == S - 1) tc_commit(bar(DL_SUM_FULL));
                    }
                    __syncwarp();
                    if (++ia == DL_NSA) { ia = 0; pa ^= 1; }
                }
            n += S;
        }
    } else if (warp == 3 || warp > DL_WB) {
        // ============================== MMA issuers: l = h1 B_d (pass 2), d = h2 B_w (pass 3) of the even / odd slices ==============================
        const int odd = warp > DL_WB;
        int n0 = 0, ib = 0, pb = 0;                          // (B ring position and its phase)
        uint32_t phases = 0;                                 // bit: parity of the set's next accumulator
        int turn = 0;                                        // slices of the other issuer so far
        int acc = 0;                                         // accumulator of slice n: a ring that both issuers' slices take in turn
        bool alive = true;
        int ti = 0;
        for (long long r = r_first; r < r_end && alive; r += 128, ++ti) {
            n0 += S;
            const int n_tile = n0;
            for (int pass = 1; pass < 3 && alive; ++pass, n0 += S) {
                if (!wait_warp(pass == 1 ? DL_H1_READY : DL_H2_READY, ti)) { alive = false; break; }
                const int kn = pass == 1 ? p.kd : p.kw;
                for (int n = n0; n < n0 + S; ++n) {
                    const int set = n & (DL_NSET - 1), before = (n - DL_NACC) & (DL_NSET - 1);
                    if ((n & 1) == odd) {
                        const int slot = odd * DL_NSB + ib;
                        // Slice n - 3 had the accumulator (the tile before had read all of its when h1 was ready).  Its set's slice before
                        // that is n - 7, which this issuer has waited for, and the one after it is n + 1, whose product waits for DL_TURN.
                        if (!wait_warp(DL_BFULL + slot, pb) || (n - DL_NACC >= n_tile && !wait_warp(DL_ACC_FREE + before, (phases >> before) + 1))) { alive = false; break; }
                        if (n > n_tile && !wait_warp(DL_TURN + 1 - odd, turn + 1)) { alive = false; break; }
                        mbar_arrive_if(bar(DL_TURN + odd), lane == 0);
                        tc_fence_after();
                        if (elect_one()) {
                            const uint64_t db = smem_desc(bstage(slot));
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                if (kk < kn) tc_mma_ta(tmem + DL_TM_ACC + 64 * acc, tmem + DL_TM_H + 8 * kk, db + (uint64_t)(128 * kk), DL_IDESC, kk > 0 ? 1u : 0u);
                            tc_commit(bar(DL_ACC_FULL + set));
                            tc_commit(bar(DL_BEMPTY + slot));
                        }
                        __syncwarp();
                        if (++ib == DL_NSB) { ib = 0; pb ^= 1; }
                    } else {
                        ++turn;
                    }
                    phases ^= 1u << set;
                    if (++acc == DL_NACC) acc = 0;
                }
            }
            if (alive && elect_one()) tc_commit(bar(DL_H_FREE));      // (all products of this warp so far)
            __syncwarp();
        }
    } else {
        // ============================== worker warps ==============================
        const int set = (warp - DL_W0) / DL_NWS;         // takes the slices n with n mod 4 == set
        const int sp = warp & 3;                         // tensor-memory sub-partition: accumulator rows 32*sp .. 32*sp+31
        const int row = 32 * sp + lane;                  // this lane's token row inside the tile
        const uint32_t tlane = tmem + ((uint32_t)(32 * sp) << 16);
        const uint32_t own_off = 128 * row, own_xor = (row & 7) << 4;
        const uint32_t up_off = row == 0 ? DL_OFF_PREV : 128 * (row - 1), up_xor = row == 0 ? 0u : ((row - 1) & 7) << 4;
        uint32_t op_phase = 1, acc_phase = 0;            // (parity of the operand's last release; of the accumulator's next arrival)
        int pending = -1;                                // x stage whose room holds an output slab that a store may still be reading
        auto release_pending = [&]() {
            if (pending >= 0) {
                if (lane == 0) bulk_wait_read<0>();
                __syncwarp();
                mbar_arrive_if(bar(DL_XEMPTY + pending), lane == 0);
                pending = -1;
            }
        };
        int ti = 0;
        bool alive = true;
        for (long long r = r_first; r < r_end && alive; r += 128, ++ti) {
            const long long tok = r + row;
            const bool live = r + 32 * sp < r_end;       // (a tile of 64 rows: two row groups only keep the barriers company)
            const bool seq_start = (tok % p.T) == 0;     // the row above belongs to another sequence: x_prev or zero
            const bool any_start = __any_sync(0xffffffffu, seq_start);
            const __nv_bfloat16* gp = (seq_start && p.x_prev && tok < p.rows) ? p.x_prev + (tok / p.T) * (long long)p.D : nullptr;
            int n0 = ti * 3 * S;
            auto acc_of = [&](int n) { return tlane + DL_TM_ACC + 64 * ((unsigned)(n - (ti + 1) * S) % DL_NACC); };     // (slices of pass 1 have none)
            // ---- passes 1 and 2: out = x + (x_above - x) * mix, mix = the pass's constants (+ l from tensor memory in pass 2).
            // The interpolation runs on packed bf16 pairs (difference, then one fused multiply-add with a single rounding):
            // its inputs and its output are bf16 anyway, and the mix is smooth in them.
#pragma unroll 1
            for (int pass = 0; pass < 2 && alive; ++pass, n0 += S) {
#pragma unroll 1
                for (int n = n0 + ((set - n0) & (DL_NSET - 1)); n < n0 + S; n += DL_NSET) {
                    const uint32_t stage = xstage(n);
                    if (!wait(DL_XFULL + (n & (DL_NSX - 1)), n / DL_NSX)) { alive = false; break; }
                    if (pass == 1) {
                        if (!wait(DL_ACC_FULL + set, acc_phase)) { alive = false; break; }
                        acc_phase ^= 1;
                        tc_fence_after();
                    }
                    __syncwarp();
                    if (!live) {
                        if (pass == 1) { tc_fence_before(); __syncwarp(); mbar_arrive_if(bar(DL_ACC_FREE + set), lane == 0); }
                        mbar_arrive_if(bar(DL_XEMPTY + (n & (DL_NSX - 1))), lane == 0);
                        if (!wait(DL_OP_FREE + set, op_phase)) { alive = false; break; }
                    } else
#pragma unroll
                    for (int hf = 0; hf < 2 && alive; ++hf) {        // 32 channels at a time (registers)
                        uint32_t mix[16];                // their mix as bf16 pairs
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            float l[16];
                            if (pass == 1) {
                                tmem_ld_row16(acc_of(n) + 32 * hf + 16 * g, l);
                            } else {
#pragma unroll
                                for (int e = 0; e < 16; ++e) l[e] = 0.f;
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const float4 v = ldsf4(stage + DL_OFF_VEC + 128 * hf + 64 * g + 16 * q);
                                mix[8 * g + 2 * q] = pack_sum(v.x, v.y, __float_as_uint(l[4 * q]), __float_as_uint(l[4 * q + 1]));
                                mix[8 * g + 2 * q + 1] = pack_sum(v.z, v.w, __float_as_uint(l[4 * q + 2]), __float_as_uint(l[4 * q + 3]));
                            }
                        }
                        if (pass == 1 && hf == 1) {      // l has been read: its accumulator is free for a later slice
                            tc_fence_before();
                            __syncwarp();
                            mbar_arrive_if(bar(DL_ACC_FREE + set), lane == 0);
                        }
#pragma unroll
                        for (int g = 2 * hf; g < 2 * hf + 2; ++g) {
                            uint4 a[2], b[2];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const uint32_t o = (uint32_t)((2 * g + q) << 4);
                                a[q] = lds128(stage + own_off + (o ^ own_xor));
                                b[q] = lds128(stage + up_off + (o ^ up_xor));
                            }
                            if (g == 3) {                // all in registers: the stage is free for a later slice
                                __syncwarp();
                                mbar_arrive_if(bar(DL_XEMPTY + (n & (DL_NSX - 1))), lane == 0);
                            }
                            if (any_start && seq_start) {
#pragma unroll
                                for (int q = 0; q < 2; ++q)
                                    b[q] = gp ? *reinterpret_cast<const uint4*>(gp + 64 * (n - n0) + 16 * g + 8 * q) : make_uint4(0u, 0u, 0u, 0u);
                            }
                            uint32_t ow[8];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const uint32_t aw[4] = {a[q].x, a[q].y, a[q].z, a[q].w}, bw[4] = {b[q].x, b[q].y, b[q].z, b[q].w};
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    uint32_t delta;
                                    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(delta) : "r"(bw[e]), "r"(aw[e]));
                                    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(ow[4 * q + e]) : "r"(delta), "r"(mix[8 * (g & 1) + 4 * q + e]), "r"(aw[e]));
                                }
                            }
                            if (g == 0) {                // the operand rows: free of the product that read them last
                                if (!wait(DL_OP_FREE + set, op_phase)) { alive = false; break; }
                                tc_fence_after();
                                __syncwarp();
                            }
                            tmem_st_row8(tlane + DL_TM_OP + 32 * set + 8 * g, ow);
                        }
                    }
                    if (!alive) break;
                    op_phase ^= 1;
                    tmem_st_done();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bar(DL_OP_READY + set), lane == 0);
                }
                if (!alive) break;
                // the pass's low-rank sum is complete: h = tanh(sum), 16 columns per set -> operand of the next products
                if (!wait(DL_SUM_FULL, pass)) { alive = false; break; }      // (two uses per tile)
                if (pass == 0 && ti > 0 && !wait(DL_H_FREE, ti - 1)) { alive = false; break; }
                tc_fence_after();
                __syncwarp();
                if (live && set < (pass == 0 ? p.kd : p.kw)) {
                    float a[16], b[16];
                    tmem_ld_row16(tlane + DL_TM_SUM + 16 * set, a);
                    if (S > 1) {
                        tmem_ld_row16(tlane + DL_TM_SUM + 64 + 16 * set, b);
#pragma unroll
                        for (int e = 0; e < 16; ++e) a[e] += b[e];
                    }
                    uint32_t ow[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) ow[e] = pack_bf16(tanh_fast(a[2 * e]), tanh_fast(a[2 * e + 1]));
                    tmem_st_row8(tlane + DL_TM_H + 8 * set, ow);
                    tmem_st_done();
                }
                tc_fence_before();
                __syncwarp();
                mbar_arrive_if(bar(pass == 0 ? DL_H1_READY : DL_H2_READY), lane == 0);
            }
            if (!alive) break;
            // ---- pass 3: d slice -> bf16, in the room of the x stage -> TMA store
#pragma unroll 1
            for (int n = n0 + ((set - n0) & (DL_NSET - 1)); n < n0 + S; n += DL_NSET) {
                const uint32_t stage = xstage(n), vec = stage + DL_OFF_VEC, slab = stage + sp * 4096;
                release_pending();
                if (!wait(DL_XFULL + (n & (DL_NSX - 1)), n / DL_NSX) || !wait(DL_ACC_FULL + set, acc_phase)) { alive = false; break; }
                acc_phase ^= 1;
                tc_fence_after();
                __syncwarp();
                if (!live) {
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bar(DL_ACC_FREE + set), lane == 0);
                    mbar_arrive_if(bar(DL_XEMPTY + (n & (DL_NSX - 1))), lane == 0);
                    continue;
                }
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    float4 v4[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) v4[q] = ldsf4(vec + 64 * g + 16 * q);
                    float v[16];
                    tmem_ld_row16(acc_of(n) + 16 * g, v);
                    if (g == 3) {
                        tc_fence_before();
                        __syncwarp();
                        mbar_arrive_if(bar(DL_ACC_FREE + set), lane == 0);
                    }
                    uint32_t o[8];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        o[2 * q] = pack_sum(v4[q].x, v4[q].y, __float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]));
                        o[2 * q + 1] = pack_sum(v4[q].z, v4[q].w, __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        sts128(slab + swz(lane, (2 * g + q) << 4), make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]));
                }
                fence_proxy_async();
                __syncwarp();
                const long long grow = r + 32 * sp;
                if (lane == 0 && grow < p.rows) {
                    tma_store_2d(&tm_d32, 64 * (n - n0), (int)grow, slab);
                    bulk_commit();
                }
                pending = n & (DL_NSX - 1);
            }
            release_pending();
        }
        if (lane == 0) bulk_wait<0>();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
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
