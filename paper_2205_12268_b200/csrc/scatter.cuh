// Dequantize + scatter + inverse transform of a layer whose contraction ran on the compressed columns (steps D and E of the WCC
// workflow; Alg. 1).
#pragma once

#include "common.cuh"
#include "patch.cuh"

namespace wcc {

// One warp per (image, tile, group of ocw output channels; ocw a multiple of 4).  rank[n][p] is the row of position p in the
// compressed matrix (or -1 when p was dropped: the zero map).  acc row r = n*k + rank holds the int32 accumulators (or fp32
// products when ACCF) of all output channels, pitch ldc (multiple of 4).  Four channels at a time: their accumulators are
// gathered while the four before are transformed, dequantized straight into the pre-scaled slots of the inverse.
template <typename T, int L, bool VEC, bool ACCF>
__global__ void __launch_bounds__(128, 4)
scatter_inv_kernel(const int32_t* __restrict__ acc, int ldc, const int32_t* __restrict__ rank, const float* __restrict__ amax_kept, float qmax,
                   const float* __restrict__ scale_w, int N, int Cout, int ocw, int H, int W, int k, T* __restrict__ y,
                   const T* residual, int relu)
{
    constexpr int U = 2;                               // channels transformed at a time
    using TT = HaarTile<L>;
    const int tiles_x = (W + TT::TW - 1) / TT::TW, tiles_y = H / TT::TH;
    const int groups = (Cout + ocw - 1) / ocw;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const long long gw = (long long)blockIdx.x * 4 + warp;
    if (gw >= (long long)N * tiles_x * tiles_y * groups) return;
    const int o_lo = (int)(gw % groups) * ocw;
    int n, ty, tx;
    tile_coords((int)(gw / groups), tiles_x, tiles_y, n, ty, tx);
    const LanePos lp = lane_positions<L>(H, W, ty, tx, lane);
    const PatchOff off = patch_off<T>(lp, W);
    const size_t P = (size_t)H * W, plane = P * sizeof(T);
    pdl_wait();
    pdl_launch();
    // Rows count inside the image; its first row is a 64-bit address and an access one 32 x 32 -> 64 bit multiply-add (an offset
    // into the whole matrix would not fit 32 bits: 17 images of 131072 kept positions x 8192 channels are 68 GiB).
    uint32_t row[8], kept = 0u;
    const uint32_t pitch = (uint32_t)ldc * 4u;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const int r = slot_ok<L>(lp, s) ? rank[(size_t)n * P + lp.pos[s]] : -1;
        row[s] = (uint32_t)max(r, 0);
        kept |= r >= 0 ? 1u << s : 0u;
    }
    uint64_t ab = reinterpret_cast<uint64_t>(acc) + ((uint64_t)n * k * ldc + o_lo) * 4;
    uint4 v[8];
    auto gather = [&]() {                              // the next four channels
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            v[s] = make_uint4(0u, 0u, 0u, 0u);
            if (kept & (1u << s)) v[s] = __ldg(reinterpret_cast<const uint4*>(ab + (uint64_t)row[s] * pitch));
        }
        ab += 16;
    };
    gather();
    float scale_a = 1.0f;
    if (!ACCF) scale_a = __fdiv_rn(*amax_kept, qmax);
    const bool coarse6 = L == 3 && ((lane / TT::CG) & 1) == 0;         // slot 6 holds a level-3 coefficient
    const int o_end = min(Cout, o_lo + ocw);
    uint64_t yo = reinterpret_cast<uint64_t>(y) + ((uint64_t)n * Cout + o_lo) * plane;
    const uint64_t rb = reinterpret_cast<uint64_t>(residual) + (uint64_t)n * Cout * plane;
    for (int o0 = o_lo; o0 < o_end; o0 += 4) {
        Raw<T> rs[4];
        if (residual) ldg_group<T, VEC, false, true, 4>(rb, plane, off, o0, Cout, rs);
        float sl[4][8];
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            float sc = 1.0f;
            if (!ACCF) sc = __fmul_rn(scale_a, __ldg(scale_w + min(o0 + d, Cout - 1)));
            // the halvings of the inverse are exact powers of two and commute with every rounding
            const float s1 = __fmul_rn(sc, 0.5f), s2 = __fmul_rn(sc, 0.25f);
            const float s6 = (L == 1) ? s1 : (coarse6 ? __fmul_rn(sc, 0.125f) : s2), s7 = (L == 1) ? s1 : s2;
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const uint32_t a = (d == 0) ? v[s].x : (d == 1) ? v[s].y : (d == 2) ? v[s].z : v[s].w;
                const float f = ACCF ? __uint_as_float(a) : __int2float_rn((int)a);
                sl[d][s] = __fmul_rn(f, s < 6 ? s1 : (s == 6 ? s6 : s7));
            }
        }
        if (o0 + 4 < o_end) gather();
#pragma unroll
        for (int h = 0; h < 4; h += U) {
            float p[U][2][4];
            inv_group<T, L, U>(*reinterpret_cast<const float(*)[U][8]>(&sl[h]), p, lane);
#pragma unroll
            for (int d = 0; d < U; ++d) {
                if (residual) {                        // the skip connection (Eq. 13): one fp32 addition per element
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        float q[4];
                        if constexpr (sizeof(T) == 4) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) q[i] = __uint_as_float(rs[h + d].w[r][i]);
                        } else {
                            q[0] = bf16lo(rs[h + d].w[r][0]); q[1] = bf16hi(rs[h + d].w[r][0]);
                            q[2] = bf16lo(rs[h + d].w[r][1]); q[3] = bf16hi(rs[h + d].w[r][1]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) p[d][r][i] = __fadd_rn(p[d][r][i], q[i]);
                    }
                }
                if (relu) relu_patch(p[d]);
                if (o0 + h + d < o_end) store_rows<T, VEC>(yo, off, lp.ok0, lp.ok1, p[d]);
                yo += plane;
            }
        }
    }
}

template <typename T, int L, bool VEC>
static wcc_status scatter_inv_dispatch(const int32_t* acc, int ldc, bool accf, const int32_t* rank, const float* amax_kept, float qmax,
                                       const float* scale_w, int N, int Cout, int H, int W, int k, void* y, const void* residual, int relu,
                                       cudaStream_t st)
{
    using TT = HaarTile<L>;
    // channels per warp: as many as still leave about 32 warps for each SM (8 to 64)
    const long long tiles = (long long)N * ceil_div(W, TT::TW) * (H / TT::TH);
    int ocw = 64;
    while (ocw > 8 && tiles * ceil_div(Cout, ocw) < B200_SMS * 32) ocw >>= 1;
    const long long warps = tiles * ceil_div(Cout, ocw);
    auto go = [&](auto kern) -> wcc_status {
        return launch_overlapped(kern, dim3((unsigned)((warps + 3) / 4)), dim3(128), 0, st, true, 1, acc, ldc, rank, amax_kept, qmax, scale_w, N, Cout,
                                 ocw, H, W, k, static_cast<T*>(y), static_cast<const T*>(residual), relu);
    };
    return accf ? go(scatter_inv_kernel<T, L, VEC, true>) : go(scatter_inv_kernel<T, L, VEC, false>);
}

wcc_status launch_scatter_inv(const int32_t* acc, int ldc, bool acc_is_float, const int32_t* rank, const float* amax_kept, int bits,
                              const float* scale_w, int N, int Cout, int H, int W, int L, int k, wcc_dtype dt, void* y, cudaStream_t st,
                              const void* residual, int relu)
{
    const bool vec = (W % 4) == 0;
    const float qmax = (bits >= 2) ? (float)((1 << (bits - 1)) - 1) : 1.0f;
    WCC_DISPATCH_TLV(scatter_inv_dispatch, dt, L, vec, acc, ldc, acc_is_float, rank, amax_kept, qmax, scale_w,
                     N, Cout, H, W, k, y, residual, relu, st);
}

}  // namespace wcc
