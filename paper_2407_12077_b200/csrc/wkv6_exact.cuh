// Token-by-token fp32 WKV-6 recurrence on the ALUs (the "exact" kernel).
//
// The value columns of a state do not interact, so a (sequence, head) unit may be cut into column slabs of 8 CW columns; and the
// recurrence over a run of tokens is an affine map of the state, S <- D S + dS with D the product of the run's decays, so the
// tokens may be cut into runs.  A cluster of G CTAs takes one slab of a unit through the sequence in rounds of G blocks of `tb`
// tokens, one block per CTA; a CTA's eight compute warps are CW column groups x NT runs of its block.  In a round every run is walked
// from a zero state first (dS and D, no outputs), every CTA publishes what its block as a whole does to a state, every run folds
// what lies before it (blocks of the cluster, through distributed shared memory, then runs of its own block) over the round's
// start state, and all runs are walked with outputs at once.  G = NT = 1 walks straight through.
// A lane has rows 4 rg .. +3 and 32 + 4 rg .. +3 of two columns (rg = lane / 4: 16 state elements in registers): r, k and w come
// as two 128-bit shared-memory loads each for 16 multiply-add pairs on row pairs (two-lane fp32), and the outputs' sum over the
// eight row groups is a transposing butterfly over four tokens and two columns, after which every lane has one output.
// Eight staging warps work one block ahead: they form w = exp(-exp(x)) and the bonus coefficient sum_i r_i u_i k_i once per
// (token, channel); fp32 inputs come by cp.async straight into the place they are read from, two blocks ahead.
// Per token
//   y_t[j] = sum_i r_t[i] (S[i][j] + u[i] k_t[i] v_t[j])      (output before the update)
//   S[i][j] = w_t[i] S[i][j] + k_t[i] v_t[j].
// D is a plain product: where it falls below 2^-100 in some channel, a large state's remainder could be lost to underflow, so
// such a fold multiplies the state by the run's decays one token after another instead.
// No atomics: results are deterministic.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "wkv6_chunked.cuh"

namespace gf {

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

constexpr int EX_N = 64;       // head size
constexpr int EX_NCW = 8;      // compute warps
constexpr int EX_NSW = 8;      // staging warps
constexpr float EX_D_MIN = 7.888609e-31f;      // 2^-100

__device__ __forceinline__ float4 ld_quad(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld_quad(const __nv_bfloat16* p)
{
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    return make_float4(ck::bf_lo(w.x), ck::bf_hi(w.x), ck::bf_lo(w.y), ck::bf_hi(w.y));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Shared memory of a CTA, in floats: two block buffers {r, k, w [TB][64], v [TB][NC], coefficient [TB]}; per run dS (in the lanes'
// layout of a compute warp; later the run's start state) and D; the same of the whole block, by parity of the round; the next round's
// start state, by parity; whether the block's D is small, by parity; abort word and wait limit; two mbarriers.
template <int CW, int NT, int TB> struct ExLayout {
    static constexpr int NC = 8 * CW;
    static constexpr int R = 0, K = TB * EX_N, W = 2 * TB * EX_N, V = 3 * TB * EX_N, COEF = V + TB * NC, BUF = COEF + TB;
    static constexpr int DS = 2 * BUF;                       // [NT][CW][4][32 lanes][4]
    static constexpr int D = DS + EX_NCW * 512;              // [NT][64]
    static constexpr int PUB = D + NT * EX_N;                // [2][CW][4][32 lanes][4]
    static constexpr int PUB_D = PUB + 2 * CW * 512;         // [2][64]
    static constexpr int S0 = PUB_D + 2 * EX_N;              // [2][CW][4][32 lanes][4]
    static constexpr int SMALL = S0 + 2 * CW * 512;          // [2] int
    static constexpr int ABORT = SMALL + 2, BAR = ABORT + 2;
    static constexpr int BYTES = (BAR + 4) * 4;
    static_assert(CW * NT == EX_NCW && BYTES <= 232448 && TB % (4 * NT) == 0 && BAR % 2 == 0, "");
};

// ---- thread-block clusters
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, int rank)      // an address of this CTA's shared memory in another CTA's
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 cluster_ld2(uint32_t a)
{
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait for a phase that other CTAs of the cluster complete.  When it runs out the status is raised and the warp goes on
// (every loop of the kernel ends by itself): later waits give up at once.
__device__ __noinline__ void cluster_mbar_wait(uint32_t bar, uint32_t parity, uint32_t abort_flag)
{
    unsigned long long t0 = 0;
    for (int n = 0;; ++n) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity), "r"(ck::TRY_WAIT_HINT_NS) : "memory");
        if (ok) return;
        if ((n & 63) != 63) continue;
        if (ck::lds32(abort_flag)) return;
        const unsigned long long now = ck::globaltimer();
        if (t0 == 0) t0 = now;
        if (now - t0 > 1000ull * ck::lds32(abort_flag + 4)) break;
        __nanosleep(64);
    }
    ck::sts32(abort_flag, 1u);
    atomicExch(&g_dev_status, 1);
}

// Meeting points of the compute warps.  They follow code in which lanes may part (a fold goes token by token where a lane's own D
// is small, a wait ends for each lane by itself), and an aligned barrier wants the whole warp at once: so the warp meets first.
__device__ __forceinline__ void ex_bar_sync()
{
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(32 * EX_NCW) : "memory");
}
__device__ __forceinline__ int ex_bar_or(int any)
{
    __syncwarp();
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %0, 0;\n\tbarrier.cta.red.or.aligned.pred q, 1, %1, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "+r"(any) : "n"(32 * EX_NCW) : "memory");
    return any;
}

// Dense: cu_seqlens == nullptr, unit = b * H + h, rows b*T .. b*T+T-1.
// Packed: unit = s * H + h, rows cu_seqlens[s] .. cu_seqlens[s+1]-1.
// Grid: units * (8 / CW) * G, clusters of G; CTA: the compute warps, then the staging warps.  tb: tokens per block, a multiple
// of 4 NT up to TB; limit_us: of a wait for the cluster (0: the default).
template <typename IO, int CW, int NT, int TB>
__global__ void __launch_bounds__(32 * (EX_NCW + EX_NSW), 1)
wkv6_exact_kernel(const IO* __restrict__ r, const IO* __restrict__ k, const IO* __restrict__ v,
                  const IO* __restrict__ x, const float* __restrict__ u,
                  const float* state_in, float* state_out, IO* __restrict__ y,
                  const int32_t* __restrict__ cu_seqlens, int T, int H, int tb, int G, uint32_t limit_us)
{
    using Lay = ExLayout<CW, NT, TB>;
    constexpr int NC = Lay::NC, NSLAB = EX_N / NC;
    extern __shared__ __align__(16) float exs[];

    const int rank = blockIdx.x % G, slab = blockIdx.x / G % NSLAB, unit = blockIdx.x / G / NSLAB;      // (rank: in the cluster)
    const int seq = unit / H, h = unit % H;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t sb = ck::smem_u32(exs), abort_flag = sb + 4 * Lay::ABORT, bar_pub = sb + 4 * Lay::BAR, bar_fold = bar_pub + 8;
    if (threadIdx.x == 0) {
        ck::mbar_init(bar_pub, G);               // every CTA's block has been published
        ck::mbar_init(bar_fold, G);              // (rounds with a small D) ... and folded by every CTA
        ck::sts32(abort_flag, 0u);
        ck::sts32(abort_flag + 4, limit_us ? limit_us : ck::WAIT_LIMIT_US);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (G > 1) { __syncwarp(); cluster_arrive(); }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    long long row0;
    int len;
    if (cu_seqlens) {
        row0 = cu_seqlens[seq];
        len = cu_seqlens[seq + 1] - cu_seqlens[seq];
    } else {
        row0 = (long long)seq * T;
        len = T;
    }
    const long long C = (long long)H * EX_N;
    const int n_blocks = (len + tb * G - 1) / (tb * G);      // rounds; this CTA's block of round b starts at token (b G + rank) tb
    const int run = tb / NT;

    if (warp < EX_NCW) {
        // ============================== compute warps ==============================
        const int cw = warp % CW, ts = warp / CW;            // column group, run
        const int rg = lane >> 2, col = 8 * cw + 2 * (lane & 3);         // this lane's first column inside the slab
        const size_t sbase = (size_t)unit * EX_N * EX_N + (size_t)(4 * rg) * EX_N + NC * slab + col;
        float2 S[2][4];                          // [column][row pair]: rows 4 rg + (0,1), (2,3), 32 + 4 rg + (0,1), (2,3)
        auto row_of = [](int i) { return (i & 1) * 2 + (i >> 1) * 32; };
        auto load_lane = [&](const float* p) {   // a state in the lanes' layout
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 f = *reinterpret_cast<const float4*>(p + 128 * q + 4 * lane);
                S[q >> 1][2 * (q & 1)] = make_float2(f.x, f.y); S[q >> 1][2 * (q & 1) + 1] = make_float2(f.z, f.w);
            }
        };
        auto store_lane = [&](float* p) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 a = S[q >> 1][2 * (q & 1)], b = S[q >> 1][2 * (q & 1) + 1];
                *reinterpret_cast<float4*>(p + 128 * q + 4 * lane) = make_float4(a.x, a.y, b.x, b.y);
            }
        };
        auto zero = [&]() {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) S[j][i] = make_float2(0.f, 0.f);
        };
        if (state_in && ts == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 a = *reinterpret_cast<const float2*>(state_in + sbase + (size_t)row_of(i) * EX_N);
                const float2 b = *reinterpret_cast<const float2*>(state_in + sbase + (size_t)(row_of(i) + 1) * EX_N);
                S[0][i] = make_float2(a.x, b.x); S[1][i] = make_float2(a.y, b.y);
            }
        } else {
            zero();
        }
        const bool split = NT > 1 || G > 1;
        if (split && ts == 0) store_lane(exs + Lay::S0 + 512 * cw);
        // after the butterfly below a lane has one token of a group of four, one of its two columns
        const bool b4 = lane & 4, b8 = lane & 8, b16 = lane & 16;
        const int my_t = (b8 ? 2 : 0) + (b16 ? 1 : 0), my_c = col + (b4 ? 1 : 0);
        IO* yp = y + (size_t)row0 * C + (size_t)h * EX_N + NC * slab + my_c;

        // one token's k, w, v as a compute lane reads them
        struct Tok { float4 ka, kb, wa, wb; float2 v; };
        auto load_tok = [&](Tok& t, const float* bk, const float* bv) {
            t.ka = *reinterpret_cast<const float4*>(bk); t.kb = *reinterpret_cast<const float4*>(bk + 32);
            t.wa = *reinterpret_cast<const float4*>(bk + Lay::W - Lay::K); t.wb = *reinterpret_cast<const float4*>(bk + Lay::W - Lay::K + 32);
            t.v = *reinterpret_cast<const float2*>(bv);
        };
        // the update with one token's k, w, v; rows as in S
        auto update = [&](const Tok& t, float2 (*D)) {
            const float2 kk[4] = {make_float2(t.ka.x, t.ka.y), make_float2(t.ka.z, t.ka.w), make_float2(t.kb.x, t.kb.y), make_float2(t.kb.z, t.kb.w)};
            const float2 ww[4] = {make_float2(t.wa.x, t.wa.y), make_float2(t.wa.z, t.wa.w), make_float2(t.wb.x, t.wb.y), make_float2(t.wb.z, t.wb.w)};
            const float2 v0 = make_float2(t.v.x, t.v.x), v1 = make_float2(t.v.y, t.v.y);
            float2 p[2][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { p[0][i] = ck::mul2(kk[i], v0); p[1][i] = ck::mul2(kk[i], v1); }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                S[0][i] = ck::fma2(ww[i], S[0][i], p[0][i]);
                S[1][i] = ck::fma2(ww[i], S[1][i], p[1][i]);
                if (D) D[i] = ck::mul2(D[i], ww[i]);
            }
        };
        // tokens t0 .. t0 + 4 n4 - 1 of the buffer, with outputs; tok: the buffer's first token
        auto walk = [&](const float* buf, int t0, int n4, int tok) {
            const float* br = buf + Lay::R + 4 * rg + t0 * EX_N;
            const float* bv = buf + Lay::V + t0 * NC + col;
            const float* bm = buf + Lay::V + (t0 + my_t) * NC + my_c;
            const float* bc = buf + Lay::COEF + t0 + my_t;
            Tok t[2];
            float4 ra[2], rb[2];
            auto load = [&](int i, int tt) {     // (a token past the run is read, inside the buffers, and not used)
                ra[i] = *reinterpret_cast<const float4*>(br + tt * EX_N); rb[i] = *reinterpret_cast<const float4*>(br + tt * EX_N + 32);
                load_tok(t[i], br + Lay::K - Lay::R + tt * EX_N, bv + tt * NC);
            };
            load(0, 0);
#pragma unroll 1
            for (int g = 0; g < n4; ++g) {
                float q[4][2];
                const float my_v = *bm, my_cf = *bc;
#pragma unroll
                for (int tt = 0; tt < 4; ++tt) {
                    const int i = tt & 1;
                    load(i ^ 1, tt + 1);
                    float2 a[2], b[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) { a[j] = ck::mul2(make_float2(ra[i].x, ra[i].y), S[j][0]); b[j] = ck::mul2(make_float2(rb[i].x, rb[i].y), S[j][2]); }
#pragma unroll
                    for (int j = 0; j < 2; ++j) { a[j] = ck::fma2(make_float2(ra[i].z, ra[i].w), S[j][1], a[j]); b[j] = ck::fma2(make_float2(rb[i].z, rb[i].w), S[j][3], b[j]); }
                    update(t[i], nullptr);
#pragma unroll
                    for (int j = 0; j < 2; ++j) { a[j] = ck::add2(a[j], b[j]); q[tt][j] = a[j].x + a[j].y; }
                }
                // sum over the eight row groups: each step halves the values (4 tokens x 2 columns) a lane carries
                float h4[4], h2[2], h1;
#pragma unroll
                for (int tt = 0; tt < 4; ++tt) h4[tt] = (b4 ? q[tt][1] : q[tt][0]) + __shfl_xor_sync(0xffffffffu, b4 ? q[tt][0] : q[tt][1], 4);
#pragma unroll
                for (int tt = 0; tt < 2; ++tt) h2[tt] = (b8 ? h4[2 + tt] : h4[tt]) + __shfl_xor_sync(0xffffffffu, b8 ? h4[tt] : h4[2 + tt], 8);
                h1 = (b16 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, b16 ? h2[0] : h2[1], 16);
                const int tk = tok + t0 + 4 * g + my_t;
                if (tk < len) yp[(size_t)tk * C] = from_f32<IO>(fmaf(my_cf, my_v, h1));
                br += 4 * EX_N; bv += 4 * NC; bm += 4 * NC; bc += 4;
            }
        };
        // Folding is per state element: thread i has elements 2 i, 2 i + 1 (two rows of a column) of every column group, in the lanes'
        // layout.  X <- D X + dS for a run of n tokens whose decays, from this thread's rows of the first token on, lie at w (in some
        // CTA's shared memory).
        const int e2 = 2 * threadIdx.x, erow = 4 * (lane >> 3) + 16 * (warp & 1) + 2 * (lane & 1) + 32 * (warp >> 1 & 1);
        auto apply = [&](float2 X, float2 D, float2 dS, uint32_t w, int n) -> float2 {
            if (D.x < EX_D_MIN || D.y < EX_D_MIN) {
#pragma unroll 1
                for (int t = 0; t < n; ++t) X = ck::mul2(X, cluster_ld2(w + 4 * t * EX_N));
                return ck::add2(X, dS);
            }
            return ck::fma2(D, X, dS);
        };
        __syncwarp();
        if (G > 1) cluster_wait();               // (the mbarriers of the cluster's CTAs are there)
        __syncthreads();
        uint32_t folds = 0;                      // rounds with a small D
        for (int b = 0; b < n_blocks; ++b) {
            const float* buf = exs + (b & 1) * Lay::BUF;
            const int tok = (b * G + rank) * tb;
            // (tokens past the end are staged as r = k = v = 0, w = 1)
            const int n4 = (min(max(len - tok - ts * run, 0), run) + 3) >> 2;
            if (split) {
                const bool publish = rank < G - 1;
                const uint32_t w_own = sb + 4 * ((b & 1) * Lay::BUF + Lay::W + erow);
                if (ts < NT - 1 || publish) {
                    zero();
                    float2 D[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) D[i] = make_float2(1.f, 1.f);
                    const float* bk = buf + Lay::K + 4 * rg + ts * run * EX_N;
                    const float* bv = buf + Lay::V + ts * run * NC + col;
#pragma unroll 1
                    for (int g = 0; g < n4; ++g, bk += 4 * EX_N, bv += 4 * NC)
#pragma unroll
                        for (int tt = 0; tt < 4; ++tt) {
                            Tok t;
                            load_tok(t, bk + tt * EX_N, bv + tt * NC);
                            update(t, D);
                        }
                    store_lane(exs + Lay::DS + 512 * warp);
                    if (cw == 0 && (lane & 3) == 0) {    // (the column groups, and the lanes of a row group, hold the same)
                        float* dp = exs + Lay::D + 64 * ts + 4 * rg;
                        *reinterpret_cast<float4*>(dp) = make_float4(D[0].x, D[0].y, D[1].x, D[1].y);
                        *reinterpret_cast<float4*>(dp + 32) = make_float4(D[2].x, D[2].y, D[3].x, D[3].y);
                    }
                }
                ex_bar_sync();
                if (G > 1) {
                    int small = 0;
                    if (publish) {                       // what the block as a whole does to a state
                        float2 Dt = make_float2(1.f, 1.f);
#pragma unroll
                        for (int c = 0; c < CW; ++c) {
                            float2 X = make_float2(0.f, 0.f);
#pragma unroll
                            for (int q = 0; q < NT; ++q) {
                                const float2 D = *reinterpret_cast<const float2*>(exs + Lay::D + 64 * q + erow);
                                X = apply(X, D, *reinterpret_cast<const float2*>(exs + Lay::DS + 512 * (q * CW + c) + e2), w_own + 4 * q * run * EX_N, run);
                                if (c == 0) Dt = ck::mul2(Dt, D);
                            }
                            *reinterpret_cast<float2*>(exs + Lay::PUB + 512 * ((b & 1) * CW + c) + e2) = X;
                        }
                        *reinterpret_cast<float2*>(exs + Lay::PUB_D + 64 * (b & 1) + erow) = Dt;      // (every row by several threads)
                        small = Dt.x < EX_D_MIN || Dt.y < EX_D_MIN;
                    }
                    small = ex_bar_or(small);
                    if (warp == 0) {
                        if (lane == 0) ck::sts32(sb + 4 * (Lay::SMALL + (b & 1)), small);
                        __syncwarp();
                        if (lane < G) cluster_mbar_arrive(cluster_addr(bar_pub, lane));
                    }
                    cluster_mbar_wait(bar_pub, b & 1, abort_flag);
                    __syncwarp();
                }
                float2 X[CW];                            // the round's start state, kept by the CTA with the last block of the round before
                {
                    const uint32_t s_now = sb + 4 * (Lay::S0 + 512 * (b & 1) * CW + e2);
                    const uint32_t a = b > 0 && rank < G - 1 ? cluster_addr(s_now, G - 1) : s_now;
#pragma unroll
                    for (int c = 0; c < CW; ++c) X[c] = cluster_ld2(a + 2048 * c);
                }
                if (G > 1) {
                    // ... then the blocks before this one, then (below) the runs
                    const uint32_t pub = sb + 4 * (Lay::PUB + 512 * (b & 1) * CW + e2), pub_d = sb + 4 * (Lay::PUB_D + 64 * (b & 1) + erow);
#pragma unroll 1
                    for (int q = 0; q < rank; ++q) {
                        const uint32_t a = cluster_addr(pub, q);
                        const float2 D = cluster_ld2(cluster_addr(pub_d, q));
                        float2 f[CW];
#pragma unroll
                        for (int c = 0; c < CW; ++c) f[c] = cluster_ld2(a + 2048 * c);
#pragma unroll
                        for (int c = 0; c < CW; ++c) X[c] = apply(X[c], D, f[c], cluster_addr(w_own, q), tb);
                    }
                    // where a D is small the fold has read that CTA's decays, which stay until every CTA is here
                    uint32_t small = 0;
                    if (lane < G - 1)
                        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(small) : "r"(cluster_addr(sb + 4 * (Lay::SMALL + (b & 1)), lane)) : "memory");
                    if (__any_sync(0xffffffffu, small != 0)) {
                        ex_bar_sync();
                        if (warp == 0 && lane < G) cluster_mbar_arrive(cluster_addr(bar_fold, lane));
                        cluster_mbar_wait(bar_fold, folds & 1, abort_flag);
                        __syncwarp();
                        ++folds;
                    }
                }
#pragma unroll
                for (int c = 0; c < CW; ++c)
#pragma unroll
                    for (int q = 0; q < NT; ++q) {
                        float2* ds = reinterpret_cast<float2*>(exs + Lay::DS + 512 * (q * CW + c) + e2);
                        const float2 f = *ds;
                        *ds = X[c];
                        if (q < NT - 1) X[c] = apply(X[c], *reinterpret_cast<const float2*>(exs + Lay::D + 64 * q + erow), f, w_own + 4 * q * run * EX_N, run);
                    }
                ex_bar_sync();
                load_lane(exs + Lay::DS + 512 * warp);
            }
            walk(buf, ts * run, n4, tok);
            if (split && ts == NT - 1 && rank == G - 1) store_lane(exs + Lay::S0 + 512 * (((b + 1) & 1) * CW + cw));
            __syncthreads();
        }
        if (split && n_blocks == 0) load_lane(exs + Lay::S0 + 512 * cw);
        if (state_out && ts == NT - 1 && rank == G - 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                *reinterpret_cast<float2*>(state_out + sbase + (size_t)row_of(i) * EX_N) = make_float2(S[0][i].x, S[1][i].x);
                *reinterpret_cast<float2*>(state_out + sbase + (size_t)(row_of(i) + 1) * EX_N) = make_float2(S[0][i].y, S[1][i].y);
            }
        }
    } else {
        // ============================== staging warps ==============================
        // thread = 4 channels of rows st / 16 + 16 i of a block, and a share of its v
        constexpr bool ASYNC = sizeof(IO) == 4;
        constexpr int SROWS = 2 * EX_NSW, NP = TB / SROWS, NV = TB * NC / 4, VT = 32 * EX_NSW;
        static_assert(NP == 2 || NP == 4 || NP == 8, "the butterfly below");
        const int st = threadIdx.x - 32 * EX_NCW, c = 4 * (st & 15), tr = st >> 4;
        const float4 u4 = *reinterpret_cast<const float4*>(u + h * EX_N + c);
        const size_t base = (size_t)row0 * C + (size_t)h * EX_N + c;
        const size_t vbase = (size_t)row0 * C + (size_t)h * EX_N + NC * slab;
        auto fetch = [&](int b) {                // fp32 inputs of block b, straight into its buffer (x where w will stand)
            if constexpr (ASYNC) {
                if (b < n_blocks) {
                    const uint32_t buf = ck::smem_u32(exs + (b & 1) * Lay::BUF);
                    const int tok = (b * G + rank) * tb, n = min(len - tok, tb);
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        const int t = tr + SROWS * i;
                        if (t < n) {
                            const size_t off = base + (size_t)(tok + t) * C;
                            const uint32_t d = buf + 4 * (t * EX_N + c);
                            cp_async16(d + 4 * Lay::W, x + off); cp_async16(d + 4 * Lay::R, r + off); cp_async16(d + 4 * Lay::K, k + off);
                        }
                    }
                    for (int e = st; e < NV; e += VT) {
                        const int t = e / (NC / 4), cc = 4 * (e % (NC / 4));
                        if (t < n) cp_async16(buf + 4 * (Lay::V + t * NC + cc), v + vbase + (size_t)(tok + t) * C + cc);
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
        };
        auto stage = [&](int b) {                // block b: from memory (or as fetched) to what the compute warps read
            float* buf = exs + (b & 1) * Lay::BUF;
            const int tok = (b * G + rank) * tb, n = min(len - tok, tb);
            float cf[NP];
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const int t = tr + SROWS * i;
                float4 *pr = reinterpret_cast<float4*>(buf + Lay::R + t * EX_N + c), *pk = reinterpret_cast<float4*>(buf + Lay::K + t * EX_N + c),
                       *pw = reinterpret_cast<float4*>(buf + Lay::W + t * EX_N + c);
                float4 r4 = z4, k4 = z4, w4 = make_float4(1.f, 1.f, 1.f, 1.f);
                if (t < n) {
                    float4 x4;
                    if constexpr (ASYNC) {
                        r4 = *pr; k4 = *pk; x4 = *pw;
                    } else {
                        const size_t off = base + (size_t)(tok + t) * C;
                        r4 = ld_quad(r + off); k4 = ld_quad(k + off); x4 = ld_quad(x + off);
                    }
                    w4 = make_float4(expf(-expf(x4.x)), expf(-expf(x4.y)), expf(-expf(x4.z)), expf(-expf(x4.w)));
                }
                if (!ASYNC || t >= n) { *pr = r4; *pk = k4; }
                *pw = w4;
                cf[i] = fmaf(r4.x * u4.x, k4.x, r4.y * u4.y * k4.y) + fmaf(r4.z * u4.z, k4.z, r4.w * u4.w * k4.w);
            }
            for (int e = st; e < NV; e += VT) {
                const int t = e / (NC / 4), cc = 4 * (e % (NC / 4));
                if (!ASYNC || t >= n)
                    *reinterpret_cast<float4*>(buf + Lay::V + t * NC + cc) = t < n ? ld_quad(v + vbase + (size_t)(tok + t) * C + cc) : z4;
            }
            // the rows' sums over the 16 lanes, halving the rows a lane carries as long as there are several
            int mine = 0, left = NP;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                if (left > 1) {
                    left >>= 1;
                    const bool up = lane & o;
#pragma unroll
                    for (int i = 0; i < NP / 2; ++i)
                        if (i < left) cf[i] = (up ? cf[i + left] : cf[i]) + __shfl_xor_sync(0xffffffffu, up ? cf[i] : cf[i + left], o);
                    mine += up ? left : 0;
                } else {
                    cf[0] += __shfl_xor_sync(0xffffffffu, cf[0], o);
                }
            }
            if ((lane & (16 / NP - 1)) == 0) buf[Lay::COEF + tr + SROWS * mine] = cf[0];
        };
        fetch(0);
        fetch(1);
        __syncwarp();
        if (G > 1) cluster_wait();
        if (n_blocks > 0) {
            if (ASYNC) asm volatile("cp.async.wait_group 1;" ::: "memory");
            stage(0);
        }
        __syncthreads();
        for (int b = 0; b < n_blocks; ++b) {     // while block b runs: stage block b + 1 (its buffer was left before block b began)
            if (b + 1 < n_blocks) {
                if (ASYNC) asm volatile("cp.async.wait_group 0;" ::: "memory");
                stage(b + 1);
            }
            __syncthreads();
            fetch(b + 2);                        // (into block b's buffer)
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (G > 1) { __syncwarp(); asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); cluster_wait(); }      // nobody reads this CTA's shared memory any more
}

template <typename IO, int CW, int NT, int TB>
inline cudaError_t launch_exact_as(long long units, int G, int tb, cudaStream_t st, const IO* r, const IO* k, const IO* v, const IO* x,
                                   const float* u, const float* state_in, float* state_out, IO* y, const int32_t* cu, int T, int H)
{
    static PerDeviceFlag attr_set;
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    if (!attr_set.is_set(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(wkv6_exact_kernel<IO, CW, NT, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, ExLayout<CW, NT, TB>::BYTES);
        if (e != cudaSuccess) return e;
        attr_set.set(dev);
    }
    return launch_pdl_cluster(wkv6_exact_kernel<IO, CW, NT, TB>, (unsigned)(units * (8 / CW) * G), 32 * (EX_NCW + EX_NSW), ExLayout<CW, NT, TB>::BYTES, G, st,
                              r, k, v, x, u, state_in, state_out, y, cu, T, H, tb, G, wait_limit_us().load(std::memory_order_relaxed));
}

// Launches the kernel over `units` (sequence, head) units.  What bounds it is the fp32 pipe of the SMs that take part (a two-lane
// multiply-add takes two of its cycles; a split walk does 5 of them per element pair instead of 3) and, for short calls, the
// latency of the steps of a round (load, decays, walk, exchange, fold, walk: 5 us at 64 tokens per CTA, 4 without a cluster).
// B200, fp32, us per call in a graph, before (one walk per column slab, 4 or 8 slabs up to 74 units) -> now:
//   4 units of 40 tokens 4.8 -> 4.2, 256 15.5 -> 6.7, 1024 55.9 -> 18.9;  8 of 256 15.8 -> 8.2;  12 of 256 15.8 -> 12.3, 1024 56.2 -> 36.6;
//   20 of 256 17.6 -> 17.5, 1024 62.6 -> 47.6;  40 of 1024 98.4 -> 76.4;  60 of 400 40.3 -> 38.0;  80 of 1024 139 -> 109;  128 of 512 71.4 -> 57.5.
// One unit per CTA and column slabs alone, before -> now: 148 of 256 38.1 -> 29.7;  256 of 256 75.8 -> 59.6, 1024 277 -> 222;
//   512 of 256 151 -> 121;  1024 of 1 38.3 -> 19.6, 256 263 -> 212;  2048 of 256 523 -> 415, in bf16 646 -> 470.  (A CTA of this form leaves the
//   split's buffers unused and has an SM to itself all the same.)
// Up to 4 tokens one walk over all columns, split / not: 1 unit of 1 token 3.01 / 2.81 (2.63 before), 4 3.02 / 2.93 (2.87), 60 3.06 / 2.95 (4.20);  of 5
//   tokens 4 units 3.02 / 3.24.
// The lines between the forms, us (slabs alone / cluster): 8 units of 70 tokens 6.3 / 6.1, 150 8.6 / 7.4;  16 of 256 12.2 / 13, 400 17.9 / 18.1,
// 1024 42 / 36.6;  20 of 400 25.5 / 25.3, 700 43.3 / 32.6;  40 of 70 9.5 / 10.8, 130 14.9 / 12.8.
template <typename IO>
inline cudaError_t launch_exact(long long units, int n_sm, cudaStream_t st, const IO* r, const IO* k, const IO* v, const IO* x,
                                const float* u, const float* state_in, float* state_out, IO* y, const int32_t* cu, int T, int H)
{
    // column slabs up to one CTA per SM, the CTA's warps over the rest of the columns and over runs of the block
    int nt = units * 8 <= n_sm ? 8 : units * 4 <= n_sm ? 4 : units * 2 <= n_sm ? 2 : 1, G = 1;
    const long long places = n_sm * 7LL / 8;       // clusters lie within one GPC, so not every SM finds a place in one
    if (units * 32 <= places) G = 4;
    else if (units * 16 <= places && T > 96) nt = 4, G = 4;
    else if (units * 8 <= places && T > 384) nt = 2, G = 4;
    else if (units * 4 <= places && T > 384) nt = 1, G = (int)(places / units < 6 ? places / units : 6);
    else if (units * 3 <= places && units * 4 > n_sm && T >= 128) nt = 1, G = 3;
    if (T <= 4) nt = 1;                            // (one group of tokens: nothing to split)
    if (G > (T + 63) / 64) G = (T + 63) / 64;
    if (G < 1) G = 1;
    // tokens per block: the sequence in as few rounds of blocks of up to 64 as it takes, in equal blocks
    const int rounds = (int)((T + 64LL * G - 1) / (64LL * G)), q = 4 * nt;
    int tb = rounds > 0 ? (int)((T + (long long)rounds * G - 1) / ((long long)rounds * G)) : q;
    tb = (tb + q - 1) / q * q;
    cudaError_t e;
    for (;;) {
        e = nt == 8 ? launch_exact_as<IO, 1, 8, 64>(units, G, tb, st, r, k, v, x, u, state_in, state_out, y, cu, T, H)
          : nt == 4 ? launch_exact_as<IO, 2, 4, 64>(units, G, tb, st, r, k, v, x, u, state_in, state_out, y, cu, T, H)
          : nt == 2 ? launch_exact_as<IO, 4, 2, 64>(units, G, tb, st, r, k, v, x, u, state_in, state_out, y, cu, T, H)
                    : launch_exact_as<IO, 8, 1, 64>(units, G, tb, st, r, k, v, x, u, state_in, state_out, y, cu, T, H);
        if (e == cudaSuccess || G == 1) return e;
        cudaGetLastError();
        G = 1;
    }
}

}  // namespace gf
