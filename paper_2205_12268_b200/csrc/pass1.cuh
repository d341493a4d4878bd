// First pass of the fused layer, and the forward transform on its own (steps A and B-norms of the WCC workflow; Eq. 3-6,
// Alg. 1): transform x in registers, build the channel norms, the per-position max |coefficient| and the selection's
// histograms; on request store the coefficients.
//
// One CTA of NW warps per (image, tile).  The warps take the boxes of NB channels in turn (box r goes to warp r % NW), loading
// the next box of theirs straight into registers while the current one is worked on.  Only the chain of fused multiply-adds
// that builds the norms (one per position, ascending channel order) runs in sequence: the eight partial sums of every lane
// travel from the warp of box r to the warp of box r + 1 through shared memory (a "token", signalled on an mbarrier), so the
// sums are the chains a single thread would build.  A slot belongs to the receiving warp; it is free again when it is
// written next, because the chain has passed through its owner since.  Where only norms and maxima are built, the transform
// runs without its halvings; one exact factor per slot at the end.  The last step (maxima over the warps, stores, histograms) is shared by the warps.
//
// Measured (B200, whole layer before -> after; the pass it replaced fed TMA rings in shared memory): 144 -> 24 bf16 37.3 -> 34.4
// us, 384 -> 512 bf16 59.4 -> 56.2, six-layer chain 393 -> 377, 24 images of C4 131 -> 125; transform, selection and inverse of
// 4 x 64 x 192 x 320 fp32 80 -> 70 (the norms no longer take a pass over the stored coefficients).
#pragma once

#include <algorithm>

#include "common.cuh"
#include "gather.cuh"
#include "patch.cuh"

namespace wcc {

struct NormsExtra {
    uint32_t* hist1;      // [N][3][2048] (round 1 first), cleared by launch_clear in the launch before, or NULL
    uint32_t* fine;       // [N][65536]: histogram of the 16 bits below the sign of every norm, cleared with hist1
    const float* Wt;      // weights to prepare in extra CTAs, or NULL
    void* Wq;
    float* scale_w;
    int Cout, kpad, bits;
};

// What a launch produces besides the norms: per-position maxima (unless no scale is taken from them), coefficients.
enum { P1_NORMS = 0, P1_MAX = 1, P1_COEF = 2 };

// DW: a depthwise 3x3 convolution (taps fp32 [C][3][3]) is applied to x first; its output never goes to memory (App. H, "a kernel
// for a fused depthwise convolution and Haar transform").
template <typename T, int L, bool VEC, int NW, int KIND, bool DW>
__global__ void __launch_bounds__(NW * 32, ((DW && NW < 8) || NW == 1) ? 12 / NW : 16 / NW)
pass1_kernel(const T* __restrict__ x, const float* __restrict__ taps, int C, int H, int W, int weight_ctas, float* __restrict__ coef, float* __restrict__ nrm2,
             float* __restrict__ amaxpos, const NormsExtra ex, int* __restrict__ status)
{
    constexpr int NB = (sizeof(T) == 2 && !DW) ? 8 : 4;       // channels of a box (32 registers of input; a convolution's input
                                                       // is loaded channel by channel, one ahead)
    constexpr int S = 8 / ((NW < 4) ? NW : 4);         // slots a warp finishes at the end
    constexpr bool MAXV = KIND != P1_NORMS;
    // Coefficients that are stored, and all behind a convolution (bound by other things), are transformed with the halvings.
    constexpr bool HALVE = KIND == P1_COEF || DW;
    using TT = HaarTile<L>;
    __shared__ float4 token[(NW > 1) ? NW : 1][2][32];          // eight sums per lane, per receiving warp
    __shared__ float fin[(NW > 1) ? NW + 1 : 1][8][32];         // maxima per warp, norms
    __shared__ uint64_t tok_bars[NW];
    using Dw = DwTile<T, L, VEC>;
    __shared__ __align__(16) float2 tap_sm[DW ? NW : 1][2][NB * 10];
    extern __shared__ __align__(16) uint8_t dw_sm[];            // DW: [NW][Dw::BYTES]
    if (KIND == P1_COEF) pdl_wait();                   // its predecessor can be anything: nothing may be read early
    pdl_launch();
    const int warp = (NW > 1) ? __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0) : 0, lane = threadIdx.x & 31;
    if ((int)blockIdx.x < weight_ctas) {
        const int o = (int)blockIdx.x * NW + warp;
        if (o < ex.Cout) weight_prep_row(ex.Wt, o, C, ex.kpad, ex.bits, ex.Wq, ex.scale_w);
        return;
    }
    const int tiles_x = (W + TT::TW - 1) / TT::TW, tiles_y = H / TT::TH;
    int n, ty, tx;
    tile_coords((int)blockIdx.x - weight_ctas, tiles_x, tiles_y, n, ty, tx);
    const LanePos lp = lane_positions<L>(H, W, ty, tx, lane);
    const size_t P = (size_t)H * W, plane = P * sizeof(T);
    const PatchOff off = patch_off<T>(lp, W);
    const uint64_t xb = reinterpret_cast<uint64_t>(x) + (uint64_t)n * C * plane;
    const int rounds = (C + NB - 1) / NB;
    // Boxes ahead: two where the registers allow it (a lone warp per tile: C4 22.4 against 23.5 us; fp32: 24 images of C4 119.8
    // against 122.2 us a layer, but with coefficients to store 69.5 against 61.4 for the transform case of pass1's header).
    constexpr int D = (!DW && (NW == 1 || (sizeof(T) == 4 && KIND != P1_COEF))) ? 2 : 1;
    Raw<T> raw[DW ? 1 : D][DW ? 1 : NB];
    uint32_t piece[DW ? Dw::CHS : 1][DW ? Dw::IT : 1][DW ? Dw::PW : 1];
    Dw dw;
    float tapv[2] = {0.0f, 0.0f};
    auto fetch_taps = [&](int r) {                     // this lane's two of the 36 taps of box r
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int e = lane + 32 * i, g = r * NB * 9 + e;
            tapv[i] = (e < NB * 9 && g < C * 9) ? __ldg(taps + g) : 0.0f;
        }
    };
    if constexpr (DW) {
        dw.init(dw_sm + warp * Dw::BYTES, H, W, ty, tx, lane);
        if (warp < rounds) {
            dw.load(xb, plane, warp * NB, C, piece);
            fetch_taps(warp);
        }
    } else
#pragma unroll
    for (int b = 0; b < D; ++b)
        if (warp + b * NW < rounds) ldg_group<T, VEC, true, true, NB>(xb, plane, off, (warp + b * NW) * NB, C, raw[b]);
    if (NW > 1) {
        if (threadIdx.x < NW) tc::mbar_init(tc::smem_u32(&tok_bars[threadIdx.x]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncthreads();
    }
    float sc[8], amax[8];
    slot_scales<L>(lane, sc);
#pragma unroll
    for (int s = 0; s < 8; ++s) amax[s] = 0.0f;
    float2 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = make_float2(0.0f, 0.0f);
    bool ok = true;
    uint32_t parity = 0;
    for (int rb = warp; rb < rounds; rb += NW * D)
#pragma unroll
    for (int b = 0; b < D; ++b) {
        const int r = rb + b * NW;
        if (r >= rounds) break;
        float o[NB][8];
        if constexpr (DW) {
            float2 ll[NB];
            float2* tp = tap_sm[warp][((r - warp) / NW) & 1];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int e = lane + 32 * i;
                if (e < NB * 9) tp[(e / 9) * 10 + e % 9] = make_float2(tapv[i], tapv[i]);
            }
            if (r + NW < rounds) fetch_taps(r + NW);
#pragma unroll
            for (int st = 0; st < NB / Dw::CHS; ++st) {
                dw.store(st & 1, piece);
                __syncwarp();
                const int cn = (st + 1 < NB / Dw::CHS) ? r * NB + (st + 1) * Dw::CHS : (r + NW) * NB;      // the channels after these
                if (st + 1 < NB / Dw::CHS || r + NW < rounds) dw.load(xb, plane, cn, C, piece);
#pragma unroll
                for (int ch = 0; ch < Dw::CHS; ++ch) {
                    const int d = st * Dw::CHS + ch;
                    float2 k[10];
                    dw_read_taps(tp + d * 10, k);
                    dw.conv(st & 1, ch, k, ll[d], o[d]);
                }
            }
            fwd_levels<L, NB, HALVE>(ll, o, lane);
        } else {
#pragma unroll
        for (int g = 0; g < NB; g += 4) fwd_group<T, L, 4, HALVE>(raw[b] + g, *reinterpret_cast<float(*)[4][8]>(&o[g]), lane);
        if (r + NW * D < rounds) {                     // the words of this box are consumed: the next box goes into their registers
            if ((r + NW * D) * NB + NB <= C) ldg_group<T, VEC, true, false, NB>(xb, plane, off, (r + NW * D) * NB, C, raw[b]);
            else ldg_group<T, VEC, true, true, NB>(xb, plane, off, (r + NW * D) * NB, C, raw[b]);
        }
        }
        if (r == rounds - 1) {                         // channels beyond the last one repeat it: they count nothing
#pragma unroll
            for (int d = 1; d < NB; ++d)
                if (r * NB + d >= C) {
#pragma unroll
                    for (int s = 0; s < 8; ++s) o[d][s] = 0.0f;
                }
        }
        if (KIND == P1_COEF) {
#pragma unroll
            for (int d = 0; d < NB; ++d) {
                if (r * NB + d < C) store_slots<L, VEC>(coef + ((size_t)n * C + r * NB + d) * P, lp, o[d]);
            }
        }
        if (MAXV) {
#pragma unroll
            for (int d = 0; d < NB; ++d)
#pragma unroll
                for (int s = 0; s < 8; ++s) amax[s] = fmaxf(amax[s], fabsf(o[d][s]));
        }
        if (NW > 1 && r > 0) {                         // the token: partial sums of the boxes before this one
            ok = ok && tc::mbar_wait(tc::smem_u32(&tok_bars[warp]), parity);
            parity ^= 1u;
            const float4 t0 = token[warp][0][lane], t1 = token[warp][1][lane];
            acc[0] = make_float2(t0.x, t0.y); acc[1] = make_float2(t0.z, t0.w);
            acc[2] = make_float2(t1.x, t1.y); acc[3] = make_float2(t1.z, t1.w);
        }
#pragma unroll
        for (int d = 0; d < NB; ++d)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 v = make_float2(o[d][2 * i], o[d][2 * i + 1]);
                acc[i] = __ffma2_rn(v, v, acc[i]);
            }
        if (NW > 1 && r + 1 < rounds) {
            const int to = (warp + 1 == NW) ? 0 : warp + 1;
            token[to][0][lane] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
            token[to][1][lane] = make_float4(acc[2].x, acc[2].y, acc[3].x, acc[3].y);
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(&tok_bars[to]));
        }
    }
    if (KIND == P1_COEF && !nrm2 && !amaxpos) return;
    // ---- the norms and maxima of the tile -------------------------------------------------------------
    float nacc[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) { nacc[2 * i] = acc[i].x; nacc[2 * i + 1] = acc[i].y; }
    if (NW > 1) {
        if (warp == (rounds - 1) % NW) {
#pragma unroll
            for (int s = 0; s < 8; ++s) fin[NW][s][lane] = nacc[s];
        }
        if (MAXV) {
#pragma unroll
            for (int s = 0; s < 8; ++s) fin[warp][s][lane] = amax[s];
        }
        __syncthreads();
    }
    pdl_wait();                                        // the histograms are cleared
    float* nr = nrm2 + (size_t)n * P;
    float* am = amaxpos + (size_t)n * P;
    auto finish = [&](int s0, auto first) {            // slots first .. first + S - 1
        constexpr int F = decltype(first)::value;
        if (s0 != F) return;
        float v[S], m[S];
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const int s = F + i;
            v[i] = (NW > 1) ? fin[NW][s][lane] : nacc[s];
            if (!HALVE) v[i] = __fmul_rn(v[i], __fmul_rn(sc[s], sc[s]));
            if (MAXV) {
                m[i] = (NW > 1) ? fin[0][s][lane] : amax[s];
#pragma unroll
                for (int w = 1; w < NW; ++w) m[i] = fmaxf(m[i], fin[w][s][lane]);
                if (!HALVE) m[i] = __fmul_rn(m[i], sc[s]);
            }
        }
#pragma unroll
        for (int i = 0; i < S; i += 2) {
            const int s = F + i;
            if (VEC && (L == 1 || s < 6)) {            // adjacent, 8-byte aligned positions
                if (lp.ok0) {
                    if (KIND != P1_COEF || nrm2) *reinterpret_cast<float2*>(nr + lp.pos[s]) = make_float2(v[i], v[i + 1]);
                    if (MAXV && amaxpos) *reinterpret_cast<float2*>(am + lp.pos[s]) = make_float2(m[i], m[i + 1]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (slot_ok<L>(lp, s + j)) {
                        if (KIND != P1_COEF || nrm2) nr[lp.pos[s + j]] = v[i + j];
                        if (MAXV && amaxpos) am[lp.pos[s + j]] = m[i + j];
                    }
                }
            }
        }
        // Norms that are exactly zero are not counted: after a ReLU whole regions of a map are zero, and their positions
        // would all hit one bin (thousands of atomics on one address).  The selection knows the number of positions, so
        // the zeros are what the bins leave out; they rank below everything else.
        if (KIND != P1_COEF && ex.hist1) {             // norms are >= +0: the digits are the bits below the sign
            uint32_t* h = ex.hist1 + (size_t)n * 3 * 2048;
            uint32_t* f = ex.fine + (size_t)n * 65536;
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const bool count = slot_ok<L>(lp, F + i) && v[i] != 0.0f;
                hist_add(h, norm_digit11(v[i]), count);
                if (count) atomicAdd(&f[norm_digit16(v[i])], 1u);      // spread out: plain atomics
            }
        }
    };
    const int s0 = warp * S;
    finish(s0, std::integral_constant<int, 0>{});
    if constexpr (NW >= 2) finish(s0, std::integral_constant<int, S>{});
    if constexpr (NW >= 4) {
        finish(s0, std::integral_constant<int, 2 * S>{});
        finish(s0, std::integral_constant<int, 3 * S>{});
    }
    if (NW > 1 && !__all_sync(0xFFFFFFFFu, ok ? 1 : 0) && lane == 0) atomicExch(status, (int)WCC_ERR_TIMEOUT);
}

// Warps per tile: eight up to two tiles per SM, four up to four, two up to eight, one up to 10.7, two up to 16, two (bf16) or four
// (fp32) up to 20, one beyond.  An SM holds sixteen warps of the kernels with several per tile and twelve tiles of one warp (168
// registers a thread), so the two steps back to two warps lie below a full wave of one-warp tiles (12 per SM) and after it.  The
// lines are measured, on whole layers of 600 drawn shapes, geometric mean of the rule's time over another choice's (worst case):
// 296 tiles and fewer, eight against four 1.00; 297 to 592, four against eight 0.93, against two 0.92; 593 to 1184, two against one
// 0.98, against four 0.97; 1185 to 1579, one against two 0.97 (1.00), against four 0.97; 1580 to 2368, two against one 0.98;
// 2369 to 2960 all within 2 % up to 100 channels.  bf16 and fp32 agree, but for fp32 with more than 100 channels, where four warps
// are 2 to 7 % faster on average from 740 tiles on and 5 % slower at worst.
template <typename T, int L, bool VEC, int KIND, bool DW>
static wcc_status pass1_launch(const void* x, const float* taps, int N, int C, int H, int W, float* coef, float* nrm2, float* amaxpos, const NormsExtra& ex,
                               cudaStream_t st)
{
    using TT = HaarTile<L>;
    const long long tiles = (long long)N * ceil_div(W, TT::TW) * (H / TT::TH);
    if (tiles > 0x7FFFFFFFLL - WCC_MAX_CHANNELS) return WCC_ERR_SHAPE;        // (blocks of a grid, those of the weights among them)
    DeviceInfo di;
    wcc_status s = device_info(di);
    if (s != WCC_OK) return s;
    const long long warps = 16LL * di.sms;
    const int nw = tiles * 4 > warps * 5 ? 1 : tiles > warps ? (sizeof(T) == 4 ? 4 : 2) : tiles * 3 > warps * 2 ? 2 : tiles * 2 > warps ? 1
                   : tiles * 4 > warps ? 2 : tiles * 8 > warps ? 4 : 8;
    auto go = [&](auto nwc) -> wcc_status {
        constexpr int w = decltype(nwc)::value;
        constexpr auto kern = pass1_kernel<T, L, VEC, w, KIND, DW>;
        constexpr int smem = DW ? w * DwTile<T, L, VEC>::BYTES : 0;
        const int wctas = ex.Wt ? ceil_div(ex.Cout, w) : 0;
        if (DW && (s = allow_smem<kern>(di.dev, smem)) != WCC_OK) return s;
        return launch_overlapped(kern, dim3((unsigned)(tiles + wctas)), dim3(w * 32), smem, st, KIND == P1_COEF || ex.hist1, 1, static_cast<const T*>(x), taps, C,
                                 H, W, wctas, coef, nrm2, amaxpos, ex, di.status);
    };
    if constexpr (!DW) {
        if (nw == 1) return go(std::integral_constant<int, 1>{});
        if (nw == 2) return go(std::integral_constant<int, 2>{});
    }
    if (nw <= 4) return go(std::integral_constant<int, 4>{});
    return go(std::integral_constant<int, 8>{});
}

template <typename T, int L, bool VEC>
static wcc_status pass1_dispatch(const void* x, const float* taps, int N, int C, int H, int W, float* coef, float* nrm2, float* amaxpos,
                                 const NormsExtra& ex, cudaStream_t st)
{
    if (taps) {
        if (coef) return pass1_launch<T, L, VEC, P1_COEF, true>(x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
        return pass1_launch<T, L, VEC, P1_MAX, true>(x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
    }
    if (coef) return pass1_launch<T, L, VEC, P1_COEF, false>(x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
    if (amaxpos) return pass1_launch<T, L, VEC, P1_MAX, false>(x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
    return pass1_launch<T, L, VEC, P1_NORMS, false>(x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
}

// First pass of the fused layer; taps: NULL, or a depthwise convolution in front.  With ex.hist1 set, launch_clear on the
// histograms must be the call before it on the stream.
static wcc_status launch_pass1(const void* x, const float* taps, int N, int C, int H, int W, int L, wcc_dtype dt, float* nrm2, float* amaxpos,
                               const NormsExtra& ex, cudaStream_t st)
{
    const bool vec = (W % 4) == 0;
    float* coef = nullptr;
    WCC_DISPATCH_TLV(pass1_dispatch, dt, L, vec, x, taps, N, C, H, W, coef, nrm2, amaxpos, ex, st);
}

// ---- coefficients alone ----------------------------------------------------------------------------
// One warp per (tile, `cpc` channels), four channels at a time, the next four in flight.  NORMS: the warp has all channels and
// builds norms and maxima as well; otherwise they are built afterwards from the stored map: free of the norms' chain, the
// channels of a few tiles spread over the whole chip.
template <typename T, int L, bool VEC, bool DW, bool NORMS>
__global__ void __launch_bounds__(128)
coef_kernel(const T* __restrict__ x, const float* __restrict__ taps, int N, int C, int H, int W, int cpc, float* __restrict__ coef,
            float* __restrict__ nrm2, float* __restrict__ amaxpos)
{
    using TT = HaarTile<L>;
    using Dw = DwTile<T, L, VEC>;
    __shared__ __align__(16) float2 tap_sm[DW ? 4 : 1][4 * 10];
    __shared__ __align__(16) uint8_t dw_sm[DW ? 4 : 1][DW ? Dw::BYTES : 16];
    pdl_wait();
    pdl_launch();
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int tiles_x = (W + TT::TW - 1) / TT::TW, tiles_y = H / TT::TH;
    const long long gw = (long long)blockIdx.x * 4 + warp;
    if (gw >= (long long)N * tiles_x * tiles_y) return;
    const int c_lo = (int)blockIdx.y * cpc, c_hi = min(C, c_lo + cpc);
    int n, ty, tx;
    tile_coords((int)gw, tiles_x, tiles_y, n, ty, tx);
    const LanePos lp = lane_positions<L>(H, W, ty, tx, lane);
    const size_t P = (size_t)H * W, plane = P * sizeof(T);
    const uint64_t xb = reinterpret_cast<uint64_t>(x) + (uint64_t)n * C * plane;
    float* out = coef + ((size_t)n * C + c_lo) * P;
    const PatchOff off = patch_off<T>(lp, W);
    Raw<T> raw[DW ? 1 : 4];
    uint32_t piece[DW ? Dw::CHS : 1][DW ? Dw::IT : 1][DW ? Dw::PW : 1];
    Dw dw;
    if constexpr (DW) {
        dw.init(dw_sm[warp], H, W, ty, tx, lane);
        dw.load(xb, plane, c_lo, C, piece);
    } else {
        ldg_group<T, VEC, true, true, 4>(xb, plane, off, c_lo, C, raw);
    }
    float nacc[8], amax[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) { nacc[s] = 0.0f; amax[s] = 0.0f; }
    for (int c = c_lo; c < c_hi; c += 4) {
        float o[4][8];
        if constexpr (DW) {
            float2 ll[4];
            __syncwarp();                              // the taps of the group before are read
            dw_stage_taps(taps, c, 4, C, tap_sm[warp], lane);
#pragma unroll
            for (int st = 0; st < 4 / Dw::CHS; ++st) {
                dw.store(st & 1, piece);
                __syncwarp();
                const int cn = c + (st + 1) * Dw::CHS;
                if (cn < c_hi) dw.load(xb, plane, cn, C, piece);
#pragma unroll
                for (int ch = 0; ch < Dw::CHS; ++ch) {
                    const int d = st * Dw::CHS + ch;
                    float2 k[10];
                    dw_read_taps(tap_sm[warp] + d * 10, k);
                    dw.conv(st & 1, ch, k, ll[d], o[d]);
                }
            }
            fwd_levels<L, 4, true>(ll, o, lane);
        } else {
            fwd_group<T, L, 4, true>(raw, o, lane);
            if (c + 4 < c_hi) {
                if (c + 8 <= C) ldg_group<T, VEC, true, false, 4>(xb, plane, off, c + 4, C, raw);
                else ldg_group<T, VEC, true, true, 4>(xb, plane, off, c + 4, C, raw);
            }
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            if (c + d < c_hi) {
                store_slots<L, VEC, true>(out, lp, o[d]);
                if (NORMS) {
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        nacc[s] = __fmaf_rn(o[d][s], o[d][s], nacc[s]);
                        amax[s] = fmaxf(amax[s], fabsf(o[d][s]));
                    }
                }
            }
            out += P;
        }
    }
    if (NORMS) {
        if (nrm2) store_slots<L, VEC>(nrm2 + (size_t)n * P, lp, nacc);
        if (amaxpos) store_slots<L, VEC>(amaxpos + (size_t)n * P, lp, amax);
    }
}

// How wcc_haar_fwd and its depthwise form split the channels of a tile.  0: pass1_kernel; 1: coefficients, norms and maxima by one
// warp; more: that many chunks, about 64 warps per SM, and the norms from the stored map.  Measured on some 500 drawn shapes
// (geometric means of pass1_kernel's time over the other's; `sparse`: the map's rows fill less than 5/8 of its tiles):
//  - rows of vectors: chunks 0.6 to 0.9, but 1.3 (fp32) and 1.6 (bf16) from four tiles per SM on with 257 channels, 1.1 and 1.7
//    from eight on with 97; one warp 1.5 up to eight channels from eight tiles per SM on;
//  - rows of 4m + 2: fp32 0.6 to 0.9 for chunks (1.2 to 1.3 from four tiles per SM and 97 channels on where the tiles are less
//    than 5/8 full) and at most 1.1 for one warp; bf16, where the element-wise accesses and the norms
//    together keep a warp busy, one warp 1.2 to 1.8 up to 16 channels, 1.05 to 1.8 up to 32 from one tile per SM on and 1.15 to
//    1.7 up to 96 from two on, chunks 1.2 to 2.3 from 97 channels on (145 channels of 17 x 36 x 146: 60 against 24 us);
//  - behind a convolution, where few warps per SM cost more, rows of vectors: one warp 1.2 to 1.4 up to 32 channels from eight
//    tiles per SM on; chunks 1.1 to 1.9 below half a tile per SM from 97 channels on in fp32 and 1.04 to 1.4 from 257 on in bf16,
//    1.05 to 1.2 with 257 from one per SM and with 97 from four per SM on; fp32 with 600 everywhere, for the second layer of a
//    block (1422 channels of 6 x 32 x 124 there 223 against about 130 us).  Rows of 4m + 2: fp32 one warp 1.2 up to 32 channels
//    from eight tiles per SM on, chunks 1.0 to 2.3 from 97 channels on; bf16 chunks 1.2 to 2.6 from 97 channels on below two
//    tiles per SM (0.9 above).
template <typename T, bool VEC>
static int channel_chunks(bool dw, long long tiles, bool sparse, int C, int sms)
{
    const bool b16 = sizeof(T) == 2, many = tiles >= 4 * sms, most = tiles >= 8 * sms;
    bool one = false, split = false;
    if (dw) {
        one = most && C <= 32 && (VEC || !b16);
        if (!VEC) split = C >= 97 && (!b16 || tiles < 2 * sms);
        else if (many) split = C >= 97;
        else if (tiles * 2 < sms) split = C >= (b16 ? 257 : 97);
        else split = (tiles >= sms && C >= 257) || (!b16 && C >= 600);
    } else if (VEC) {
        one = most && C <= 8;
        split = (many && C >= 257) || (most && C >= 97);
    } else if (b16) {
        one = C <= 16 || (C <= 32 && tiles >= sms) || (C <= 96 && tiles >= 2 * sms);
        split = C >= 97;
    } else {
        split = sparse && many && C >= 97;
    }
    if (one) return 1;
    return split ? (int)std::min<long long>(ceil_div(C, 4), (64LL * sms + tiles - 1) / tiles) : 0;
}

template <typename T, int L, bool VEC, bool DW>
static wcc_status coef_launch(const void* x, const float* taps, int N, int C, int H, int W, long long tiles, int chunks, float* coef, float* nrm2, float* amaxpos,
                              cudaStream_t st)
{
    const int cpc = ceil_div(ceil_div(C, chunks), 4) * 4;
    auto go = [&](auto kern) {
        return launch_overlapped(kern, dim3((unsigned)((tiles + 3) / 4), (unsigned)ceil_div(C, cpc)), dim3(128), 0, st, true, 1, static_cast<const T*>(x), taps, N,
                                 C, H, W, cpc, coef, nrm2, amaxpos);
    };
    if (chunks == 1) return go(coef_kernel<T, L, VEC, DW, true>);
    const wcc_status s = go(coef_kernel<T, L, VEC, DW, false>);
    return s != WCC_OK ? s : launch_coef_norms(coef, N, C, (long long)H * W, nrm2, amaxpos, st);
}

template <typename T, int L, bool VEC>
static wcc_status haar_fwd_dispatch(const void* x, const float* taps, int N, int C, int H, int W, float* coef, float* nrm2, float* amaxpos, cudaStream_t st)
{
    using TT = HaarTile<L>;
    const long long tiles = (long long)N * ceil_div(W, TT::TW) * (H / TT::TH);
    if (tiles > 0x7FFFFFFFLL) return WCC_ERR_SHAPE;
    DeviceInfo di;
    wcc_status s = device_info(di);
    if (s != WCC_OK) return s;
    const int chunks = channel_chunks<T, VEC>(taps != nullptr, tiles, W * 8LL < 5LL * ceil_div(W, TT::TW) * TT::TW, C, di.sms);
    if (!chunks) return pass1_dispatch<T, L, VEC>(x, taps, N, C, H, W, coef, nrm2, amaxpos, NormsExtra{}, st);
    return taps ? coef_launch<T, L, VEC, true>(x, taps, N, C, H, W, tiles, chunks, coef, nrm2, amaxpos, st)
                : coef_launch<T, L, VEC, false>(x, taps, N, C, H, W, tiles, chunks, coef, nrm2, amaxpos, st);
}

// Forward transform with stored coefficients, after the depthwise convolution if taps are given; nrm2 and amaxpos may be NULL.
wcc_status launch_haar_fwd(const void* x, const float* taps, int N, int C, int H, int W, int L, wcc_dtype dt, float* coef, float* nrm2,
                           float* amaxpos, cudaStream_t st)
{
    const bool vec = (W % 4) == 0;                     // always true for L >= 2
    WCC_DISPATCH_TLV(haar_fwd_dispatch, dt, L, vec, x, taps, N, C, H, W, coef, nrm2, amaxpos, st);
}

}  // namespace wcc
