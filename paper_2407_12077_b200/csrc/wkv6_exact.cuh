// Token-by-token fp32 WKV-6 recurrence on the ALUs (the "exact" kernel).
//
// The value columns of a state do not interact, so a (sequence, head) unit may be cut into column slabs.  A compute warp
// owns 2 CPL columns: lane = 2 rg + cl has rows 4 rg .. 4 rg + 3 of CPL columns (4 CPL state elements in registers for the
// life of the sequence); a CTA holds NCW compute warps and EX_NSW staging warps.  The recurrence is one multiply-add deep
// per token; what bounds the kernel is the instructions a scheduler issues per token, so the compute warps do nothing
// else: r, k and w of the four rows come as one 128-bit shared-memory load each, the arithmetic runs on row pairs
// (two-lane fp32), and the outputs' sum over the 16 row groups is a transposing butterfly over four tokens (and two
// columns) at once.  The staging warps work one tile of 16 tokens ahead (global loads three tiles ahead, in registers):
// they widen the inputs, form w = exp(-exp(x)) and the bonus coefficient sum_i r_i u_i k_i once per (token, channel), and
// send the outputs of the tile before to memory.  Two tile buffers, one block barrier per tile.  Per token
//   y_t[j] = sum_i r_t[i] (S[i][j] + u[i] k_t[i] v_t[j])      (output before the update)
//   S[i][j] = w_t[i] S[i][j] + k_t[i] v_t[j].
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
constexpr int EX_TT = 16;      // tokens per shared-memory tile
constexpr int EX_NSW = 8;      // staging warps (4: the exponentials of a tile take longer than its recurrence; 16: too many to schedule)

template <typename IO> __device__ __forceinline__ float2 ld_pair(const IO* p);
template <> __device__ __forceinline__ float2 ld_pair<float>(const float* p) { return *reinterpret_cast<const float2*>(p); }
template <> __device__ __forceinline__ float2 ld_pair<__nv_bfloat16>(const __nv_bfloat16* p)
{
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}
template <typename IO> __device__ __forceinline__ void st_pair(IO* p, float2 v);
template <> __device__ __forceinline__ void st_pair<float>(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
template <> __device__ __forceinline__ void st_pair<__nv_bfloat16>(__nv_bfloat16* p, float2 v)
{
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
}

// Dense: cu_seqlens == nullptr, unit = b * H + h, rows b*T .. b*T+T-1.
// Packed: unit = s * H + h, rows cu_seqlens[s] .. cu_seqlens[s+1]-1.
// Grid: units * (64 / (2 CPL NCW)); CTA: NCW compute warps, then EX_NSW staging warps.
template <typename IO, int NCW, int CPL>
__global__ void __launch_bounds__(32 * (NCW + EX_NSW))
wkv6_exact_kernel(const IO* __restrict__ r, const IO* __restrict__ k, const IO* __restrict__ v,
                  const IO* __restrict__ x, const float* __restrict__ u,
                  const float* state_in, float* state_out, IO* __restrict__ y,
                  const int32_t* __restrict__ cu_seqlens, int T, int H)
{
    constexpr int NC = 2 * CPL * NCW;            // value columns of this CTA
    constexpr int NSLAB = EX_N / NC;
    __shared__ __align__(16) float rs[2][EX_TT][EX_N], ks[2][EX_TT][EX_N], ws[2][EX_TT][EX_N], vs[2][EX_TT][NC];
    __shared__ __align__(16) float ys[2][EX_TT][NC];
    __shared__ float coef[2][EX_TT];

    const int unit = blockIdx.x / NSLAB, slab = blockIdx.x % NSLAB;
    const int seq = unit / H, h = unit % H;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
    const int n_tiles = (len + EX_TT - 1) / EX_TT;

    if (warp < NCW) {
        // ============================== compute warps ==============================
        const int rg = lane >> 1, col = CPL * (2 * warp + (lane & 1));       // this lane's first column inside the slab
        const size_t sbase = (size_t)unit * EX_N * EX_N + (size_t)(4 * rg) * EX_N + NC * slab + col;
        float S[CPL][4];                         // [column][row]
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) S[j][i] = state_in ? state_in[sbase + (size_t)i * EX_N + j] : 0.f;
        // the lane's place in the butterfly below: it ends with one token of a group of four (and one of two columns)
        const bool b2 = lane & 2, b4 = lane & 4, b8 = lane & 8;
        const int my_t = CPL == 2 ? (b4 ? 2 : 0) + (b8 ? 1 : 0) : (b2 ? 2 : 0) + (b4 ? 1 : 0);
        const int my_c = col + (CPL == 2 && b2 ? 1 : 0);
        __syncthreads();
        for (int i = 0; i < n_tiles; ++i) {
            const int b = i & 1;
#pragma unroll 2
            for (int t0 = 0; t0 < EX_TT; t0 += 4) {    // (tokens past the end are staged as r = k = v = 0, w = 1)
                float q[4][CPL];
                const float my_v = vs[b][t0 + my_t][my_c], my_cf = coef[b][t0 + my_t];
#pragma unroll
                for (int tt = 0; tt < 4; ++tt) {
                    const int t = t0 + tt;
                    const float4 r4 = *reinterpret_cast<const float4*>(&rs[b][t][4 * rg]);
                    const float4 k4 = *reinterpret_cast<const float4*>(&ks[b][t][4 * rg]);
                    const float4 w4 = *reinterpret_cast<const float4*>(&ws[b][t][4 * rg]);
                    const float2 r01 = make_float2(r4.x, r4.y), r23 = make_float2(r4.z, r4.w);
                    const float2 k01 = make_float2(k4.x, k4.y), k23 = make_float2(k4.z, k4.w);
                    const float2 w01 = make_float2(w4.x, w4.y), w23 = make_float2(w4.z, w4.w);
#pragma unroll
                    for (int j = 0; j < CPL; ++j) {
                        const float vj = vs[b][t][col + j];
                        const float2 v2 = make_float2(vj, vj);
                        float2 s01 = make_float2(S[j][0], S[j][1]), s23 = make_float2(S[j][2], S[j][3]);
                        const float2 a = ck::fma2(r23, s23, ck::mul2(r01, s01));
                        s01 = ck::fma2(w01, s01, ck::mul2(k01, v2)); s23 = ck::fma2(w23, s23, ck::mul2(k23, v2));
                        S[j][0] = s01.x; S[j][1] = s01.y; S[j][2] = s23.x; S[j][3] = s23.y;
                        q[tt][j] = a.x + a.y;
                    }
                }
                // sum over the 16 row groups: each of the first steps halves the values (4 tokens x CPL columns) a lane carries
                float h4[4], h2[2], h1;
                if constexpr (CPL == 2) {
#pragma unroll
                    for (int tt = 0; tt < 4; ++tt) h4[tt] = (b2 ? q[tt][1] : q[tt][0]) + __shfl_xor_sync(0xffffffffu, b2 ? q[tt][0] : q[tt][1], 2);
                } else {
#pragma unroll
                    for (int tt = 0; tt < 4; ++tt) h4[tt] = q[tt][0];
                }
                constexpr int M2 = 2 * CPL;
                const bool s4 = CPL == 2 ? b4 : b2, s2 = CPL == 2 ? b8 : b4;
#pragma unroll
                for (int tt = 0; tt < 2; ++tt) h2[tt] = (s4 ? h4[2 + tt] : h4[tt]) + __shfl_xor_sync(0xffffffffu, s4 ? h4[tt] : h4[2 + tt], M2);
                h1 = (s2 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, s2 ? h2[0] : h2[1], 2 * M2);
#pragma unroll
                for (int o = 4 * M2; o < 32; o <<= 1) h1 += __shfl_xor_sync(0xffffffffu, h1, o);
                if (lane < 4 * M2) ys[b][t0 + my_t][my_c] = fmaf(my_cf, my_v, h1);
            }
            __syncthreads();
        }
        if (state_out) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < CPL; ++j) state_out[sbase + (size_t)i * EX_N + j] = S[j][i];
        }
    } else {
        // ============================== staging warps ==============================
        const int sw = warp - NCW, st = threadIdx.x - 32 * NCW;
        const int c = 2 * lane;                  // this lane's channel pair
        const float2 u2 = *reinterpret_cast<const float2*>(u + h * EX_N + c);
        const bool my_v = (unsigned)(c - NC * slab) < (unsigned)NC;
        constexpr int NP = EX_TT / EX_NSW;       // tokens per staging warp and tile
        struct Raw { float2 r[NP], k[NP], v[NP], x[NP]; };
        Raw raw0, raw1;                          // two tiles as they come from memory, ahead of the one being staged
        auto fetch_tile = [&](int i, Raw& raw) {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const int t = i * EX_TT + p * EX_NSW + sw;
                if (t < len) {
                    const size_t off = (size_t)(row0 + t) * C + (size_t)h * EX_N + c;
                    raw.r[p] = ld_pair<IO>(r + off); raw.k[p] = ld_pair<IO>(k + off); raw.x[p] = ld_pair<IO>(x + off);
                    if (my_v) raw.v[p] = ld_pair<IO>(v + off);
                }
            }
        };
        auto stage_tile = [&](int i, const Raw& raw) {
            const int b = i & 1;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const int t = p * EX_NSW + sw;
                float2 rr = make_float2(0.f, 0.f), kk = rr, vv = rr, ww = make_float2(1.f, 1.f);
                if (i * EX_TT + t < len) {
                    rr = raw.r[p]; kk = raw.k[p]; vv = raw.v[p];
                    ww = make_float2(expf(-expf(raw.x[p].x)), expf(-expf(raw.x[p].y)));
                }
                *reinterpret_cast<float2*>(&rs[b][t][c]) = rr;
                *reinterpret_cast<float2*>(&ks[b][t][c]) = kk;
                *reinterpret_cast<float2*>(&ws[b][t][c]) = ww;
                if (my_v) *reinterpret_cast<float2*>(&vs[b][t][c - NC * slab]) = vv;
                // bonus coefficient sum_i r[i] u[i] k[i] of this token
                float cf = fmaf(rr.x * u2.x, kk.x, rr.y * u2.y * kk.y);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) cf += __shfl_xor_sync(0xffffffffu, cf, o);
                if (lane == 0) coef[b][t] = cf;
            }
        };
        auto write_out = [&](int i) {            // y of a tile, coalesced over its columns
            const int b = i & 1;
#pragma unroll
            for (int e = st; e < EX_TT * NC / 2; e += 32 * EX_NSW) {
                const int t = e / (NC / 2), cc = 2 * (e % (NC / 2));
                if (i * EX_TT + t < len)
                    st_pair<IO>(y + (size_t)(row0 + i * EX_TT + t) * C + (size_t)h * EX_N + NC * slab + cc,
                                *reinterpret_cast<const float2*>(&ys[b][t][cc]));
            }
        };
        if (n_tiles > 0) fetch_tile(0, raw0);
        if (n_tiles > 1) fetch_tile(1, raw1);
        if (n_tiles > 0) stage_tile(0, raw0);
        if (n_tiles > 2) fetch_tile(2, raw0);
        __syncthreads();
        auto step = [&](int i, Raw& raw) {       // while tile i runs: stage tile i + 1 from raw, which then takes tile i + 3
            if (i + 1 < n_tiles) {
                stage_tile(i + 1, raw);
                if (i + 3 < n_tiles) fetch_tile(i + 3, raw);
            }
            if (i > 0) write_out(i - 1);
            __syncthreads();
        };
        for (int i = 0; i < n_tiles; i += 2) {
            step(i, raw1);
            if (i + 1 < n_tiles) step(i + 1, raw0);
        }
        if (n_tiles > 0) write_out(n_tiles - 1);
    }
}

// Launches the kernel over `units` (sequence, head) units, cut into as many column slabs as leave no SM a second CTA: a
// slab stages r, k, w again, which costs nothing on an idle SM and everything on a busy one.  Measured in us (B200, fp32)
// with 8 / 4 / 1 slabs per unit, and with the former one-CTA-per-unit kernel (no staging warps, four-way sums):
//   4 units of 256 tokens 15.4 / 17.0 / 36.5 (53.6);  20 of 300 26.3 / 20.2 / 43.0 (63.0);
//   60 of 512 82 / 50.8 / 71.3 (107);  128 of 512 154 / 98.8 / 72.0 (108);  1024 of 256 575 / 340 / 259 (279).
template <typename IO>
inline cudaError_t launch_exact(long long units, int n_sm, cudaStream_t st, const IO* r, const IO* k, const IO* v, const IO* x,
                                const float* u, const float* state_in, float* state_out, IO* y, const int32_t* cu, int T, int H)
{
    if (units * 8 <= n_sm)
        wkv6_exact_kernel<IO, 4, 1><<<(unsigned)(units * 8), 32 * (4 + EX_NSW), 0, st>>>(r, k, v, x, u, state_in, state_out, y, cu, T, H);
    else if (units * 2 <= n_sm)                  // (up to two CTAs of 4 slabs an SM are still ahead of one whole unit)
        wkv6_exact_kernel<IO, 4, 2><<<(unsigned)(units * 4), 32 * (4 + EX_NSW), 0, st>>>(r, k, v, x, u, state_in, state_out, y, cu, T, H);
    else
        wkv6_exact_kernel<IO, 16, 2><<<(unsigned)units, 32 * (16 + EX_NSW), 0, st>>>(r, k, v, x, u, state_in, state_out, y, cu, T, H);
    return cudaGetLastError();
}

}  // namespace gf
