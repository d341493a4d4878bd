// Gather + quantization of the kept columns straight from the input (no stored coefficient map): the path of layers
// whose channel counts exceed one operand tile of the fused kernels (Alg. 1, steps A-B of the kept columns only).
#pragma once

#include "common.cuh"
#include "gather.cuh"
#include "patch.cuh"

namespace wcc {

// One warp per (image, tile, chunk of 16 / 8 channels) transforms its channels of x again (as the first pass did, after the
// depthwise convolution when DW) and writes, for every slot of the lane whose position is kept, that chunk of the position's
// row (rank[n][p] = row of position p inside image n, or -1).  Same codes as gather_quant_kernel.  All of a chunk's loads are
// in flight before the selection's results are waited for.
template <typename T, int L, bool VEC, bool QUANT, bool DW>
__global__ void __launch_bounds__(128)
regather_quant_kernel(const T* __restrict__ x, const float* __restrict__ taps, const int32_t* __restrict__ rank,
                      const float* __restrict__ amax_kept, int N, int C, int H, int W, int k, int kpad, float qmax, int clamp, void* __restrict__ Xq)
{
    using TT = HaarTile<L>;
    constexpr int CH = QUANT ? 16 : 8;                 // channels per 16-byte store
    constexpr float MAGIC = 12582912.0f;               // 1.5 * 2^23: adding it rounds to the nearest integer, ties to even
    using Dw = DwTile<T, L, VEC>;
    __shared__ __align__(16) float2 tap_sm[DW ? 4 : 1][CH * 10];
    __shared__ __align__(16) uint8_t dw_sm[DW ? 4 : 1][DW ? Dw::BYTES : 16];
    const int tiles_x = (W + TT::TW - 1) / TT::TW, tiles_y = H / TT::TH;
    const int chunks = kpad / CH;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const long long gw = (long long)blockIdx.x * 4 + warp;
    if (gw >= (long long)N * tiles_x * tiles_y * chunks) return;
    const int chunk = (int)(gw % chunks), c0 = chunk * CH;
    int n, ty, tx;
    tile_coords((int)(gw / chunks), tiles_x, tiles_y, n, ty, tx);
    const LanePos lp = lane_positions<L>(H, W, ty, tx, lane);
    const size_t P = (size_t)H * W, plane = P * sizeof(T);
    const uint64_t xb = reinterpret_cast<uint64_t>(x) + (uint64_t)n * C * plane;
    constexpr int NB = (sizeof(T) == 2) ? 8 : 4;       // channels loaded at once: 32 registers
    Raw<T> raw[DW ? 1 : NB];
    uint32_t piece[DW ? Dw::CHS : 1][DW ? Dw::IT : 1][DW ? Dw::PW : 1];
    Dw dw;
    PatchOff off;
    if constexpr (DW) {
        dw.init(dw_sm[warp], H, W, ty, tx, lane);
        dw.load(xb, plane, c0, C, piece);
        dw_stage_taps(taps, c0, CH, C, tap_sm[warp], lane);
    } else {
        off = patch_off<T>(lp, W);
        ldg_group<T, VEC, true, true, NB>(xb, plane, off, c0, C, raw);
    }
    pdl_wait();
    pdl_launch();
    int rk[8];
    bool any = false;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        rk[s] = slot_ok<L>(lp, s) ? rank[(size_t)n * P + lp.pos[s]] : -1;
        any = any || rk[s] >= 0;
    }
    if (!__any_sync(0xFFFFFFFFu, any ? 1 : 0)) return;                // nothing kept in this tile
    float mul[8];
    slot_scales<L>(lane, mul);                  // the halvings of the transform and the quantizer's factor in one
    if (DW) {                                          // (behind a convolution the transform halves, as in the first pass)
#pragma unroll
        for (int s = 0; s < 8; ++s) mul[s] = 1.0f;
    }
    if (QUANT) {
        const float amax = *amax_kept;
        const float inv = (amax > 0.0f) ? __fdiv_rn(qmax, amax) : 0.0f;
#pragma unroll
        for (int s = 0; s < 8; ++s) mul[s] = __fmul_rn(mul[s], inv);
    }
    uint32_t packed[8][4];
#pragma unroll
    for (int g = 0; g < CH / 4; ++g) {
        float o[4][8];
        if constexpr (DW) {
            float2 ll[4];
#pragma unroll
            for (int st = 0; st < 4 / Dw::CHS; ++st) {
                const int i = g * 4 + st * Dw::CHS;
                dw.store(st & 1, piece);
                __syncwarp();
                if (i + Dw::CHS < CH) dw.load(xb, plane, c0 + i + Dw::CHS, C, piece);
#pragma unroll
                for (int ch = 0; ch < Dw::CHS; ++ch) {
                    float2 kk[10];
                    dw_read_taps(&tap_sm[warp][(i + ch) * 10], kk);
                    dw.conv(st & 1, ch, kk, ll[st * Dw::CHS + ch], o[st * Dw::CHS + ch]);
                }
            }
            fwd_levels<L, 4, true>(ll, o, lane);
        } else {
            fwd_group<T, L, 4>(raw + (g * 4) % NB, o, lane);
            if ((g * 4 + 4) % NB == 0 && g * 4 + 4 < CH) ldg_group<T, VEC, true, true, NB>(xb, plane, off, c0 + g * 4 + 4, C, raw);
        }
        uint32_t code[4][8];
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const bool real = c0 + g * 4 + d < C;      // channels of the padding are zero
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                float v = __fmul_rn(o[d][s], mul[s]);
                if (QUANT) {
                    if (clamp) v = fminf(fmaxf(v, -qmax), qmax);       // a given clipping parameter can be exceeded
                    v = __fadd_rn(v, MAGIC);           // the low byte is the two's complement code of rint(v)
                }
                code[d][s] = real ? __float_as_uint(v) : 0u;
            }
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            if (QUANT) {
                packed[s][g] = __byte_perm(__byte_perm(code[0][s], code[1][s], 0x0040), __byte_perm(code[2][s], code[3][s], 0x0040), 0x5410);
            } else {
                packed[s][2 * g] = pack_bf16x2(__uint_as_float(code[0][s]), __uint_as_float(code[1][s]));
                packed[s][2 * g + 1] = pack_bf16x2(__uint_as_float(code[2][s]), __uint_as_float(code[3][s]));
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        if (rk[s] >= 0) {
            char* row = static_cast<char*>(Xq) + ((size_t)n * k + rk[s]) * kpad * (QUANT ? 1 : 2);
            *reinterpret_cast<uint4*>(row + (size_t)chunk * 16) = make_uint4(packed[s][0], packed[s][1], packed[s][2], packed[s][3]);
        }
    }
}

template <typename T, int L, bool VEC>
static wcc_status regather_dispatch(const void* x, const float* taps, const int32_t* rank, const float* amax_kept, int N, int C, int H, int W,
                                    int k, int kpad, int bits, int clamp, void* Xq, cudaStream_t st)
{
    using TT = HaarTile<L>;
    const float qmax = (bits >= 2) ? (float)((1 << (bits - 1)) - 1) : 1.0f;
    const long long warps = (long long)N * ceil_div(W, TT::TW) * (H / TT::TH) * (kpad / (bits >= 2 ? 16 : 8));
    if (warps > 0x7FFFFFFFLL * 4) return WCC_ERR_SHAPE;
    auto go = [&](auto kern) -> wcc_status {
        return launch_overlapped(kern, dim3((unsigned)((warps + 3) / 4)), dim3(128), 0, st, true, 1, static_cast<const T*>(x), taps, rank, amax_kept, N, C,
                                 H, W, k, kpad, qmax, clamp, Xq);
    };
    if (taps) return bits >= 2 ? go(regather_quant_kernel<T, L, VEC, true, true>) : go(regather_quant_kernel<T, L, VEC, false, true>);
    return bits >= 2 ? go(regather_quant_kernel<T, L, VEC, true, false>) : go(regather_quant_kernel<T, L, VEC, false, false>);
}

// taps: NULL, or the depthwise convolution that the first pass applied.  The kernel before it on the stream is the selection of
// the same layer (or follows it): x is read before that is waited for.
wcc_status launch_regather_quant(const void* x, const float* taps, const int32_t* rank, const float* amax_kept, int N, int C, int H, int W, int L,
                                 int k, int kpad, int bits, bool clamp, wcc_dtype dt, void* Xq, cudaStream_t st)
{
    const bool vec = (W % 4) == 0;
    WCC_DISPATCH_TLV(regather_dispatch, dt, L, vec, x, taps, rank, amax_kept, N, C, H, W, k, kpad, bits, (int)clamp, Xq, st);
}

}  // namespace wcc
