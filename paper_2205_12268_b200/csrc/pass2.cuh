// Second pass of the fused layer (steps A, C, D, E of the WCC workflow, Eq. 9 / Alg. 1, with the index set and the
// activation scale of step B already known): transform from x, keep / drop, quantize, pointwise convolution on tensor
// cores, dequantize, inverse transform, store y.  Neither the coefficient map, nor the compressed matrix, nor the
// accumulators, nor the zero-filled map ever reach HBM.
//
// A CTA owns four warp tiles (4 x 256 = 1024 wavelet-domain positions, see haar.cuh) and runs 4 * WPT warps.  Warp w works
// for tile t = w % 4; the WPT warps of a tile split the input channels (in units of eight) on the way in and the output
// channels (in groups of four) on the way out.  Rows of the A operand are ordered  slot * 128 + t * 32 + lane,  so MMA
// block b (128 rows) holds slot b of all four tiles and the accumulators of tile t's lanes sit in TMEM lanes 32t .. 32t+31:
// exactly the lane quarter that warp w = t (mod 4) may read.  Every thread therefore reads back its own eight slots of an
// output channel with tcgen05.ld and runs the inverse transform in registers; nothing is transposed through shared memory.
//
// Inputs go from global memory straight into registers, a batch of channels ahead of the one being transformed: a lane's
// patch of a channel is one vector load per row, so a staging ring in shared memory only added instructions (a wait, a
// refill and two shared loads per patch) and took the shared memory that now holds the A operand.  Phases are separated by
// block barriers; what one CTA waits for, the other CTA on the SM (WPT = 2) or the other twelve warps (WPT = 4) cover.
// The A operand holds all K of a layer, or one of several K parts that are accumulated in turn; output channels go through
// TMEM in chunks of `nchunk`.  The one mbarrier wait is bounded and reports WCC_ERR_TIMEOUT.
//
// Measured (B200, back-to-back calls) against the kernels it replaced (TMA rings, one CTA of nine warps per SM; one tile per
// CTA for the shapes beyond that): C4 fp32 43.4 -> 36.5 us (x and y cross HBM once each: 5.2 TB/s, 79 % of the copy rate),
// 24 images of it 77.7 -> 71.4; 24 -> 144 channels bf16 unquantized on 2 x 256 x 512 34.3 -> 22.8; 32 -> 192 there
// 46.6 -> 30.2; 96 -> 96 with residual, ReLU and clipping on 4 x 128 x 256 63.2 -> 23.3.  Both types wait: half
// (bf16) to two thirds (fp32) of the issue slots are free, at sixteen warps per SM.
#pragma once

#include "common.cuh"
#include "contract.cuh"
#include "patch.cuh"

namespace wcc {
namespace p2 {

constexpr int TILES = 4;                    // warp tiles per CTA
constexpr int ROWS = TILES * 256;           // operand rows per CTA
constexpr float MAGIC = 12582912.0f;        // 1.5 * 2^23: adding it rounds to the nearest integer, ties to even

struct Ctl {
    uint64_t done;                          // tcgen05.commit of the instructions issued so far
    uint32_t tmem_base;
    int pad;
};

struct Params {
    const void* x; const uint8_t* Wq; const int32_t* rank; const float* nrm2; const uint32_t* thr; const float* amax_kept;
    const float* scale_w; float qmax;
    float alpha;                 // > 0: given clipping parameter of the activation quantizer (codes are clamped)
    int relu;                    // non-zero: y = max(., 0)
    const void* residual;        // NULL, or [N][Cout][H][W] of the activation type, added before the ReLU
    int N, Cin, Cout, H, W, k, krow, npad, nchunk, ksteps_part, b_resident, tmem_cols, tiles_total;
    int grp0;                    // the launch's first tile group
    int split_from, parts, share;    // CTAs from split_from on share a tile group `parts` ways, `share` output channels each
    int followed;                // non-zero (WPT = 2 only): a launch for the last groups of the layer comes behind this one
    int last;                    // non-zero (WPT = 4 only): that launch
    uint32_t* selected;          // zero until a CTA of a launch with `followed` has waited for the selection
    void* y; uint8_t* xq_tap; int32_t* acc_tap; int* status;
};

__device__ __forceinline__ uint64_t smem_desc_plain(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    const uint32_t lo = ((addr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
    const uint32_t hi = (sbo_bytes >> 4) | (1u << 14);      // version 1, layout type 0 (no swizzle)
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr));
}

// MODE is a set of compiled-in features: 1 = ReLU on the way out, 2 = taps for tests, 4 = a given clipping parameter (codes
// are clamped), 8 = residual add.  A compiled-in feature is still switched by its run-time argument; a feature that is not
// compiled in costs nothing (as run-time branches in one kernel the options cost the plain layer 7-18 %).
// Instantiated: 0 (plain), 1, 13 and 15 (everything); a request runs on the smallest variant that contains it.  Taps run with
// WPT = 4 only, and so do maps with W = 4m + 2, plain or with everything.
template <typename T, int L, bool I8, int WPT, bool VEC, int MODE>
__global__ void __launch_bounds__(TILES * WPT * 32, WPT == 2 ? 2 : 1)
pass2_kernel(const Params pr)
{
    constexpr bool RELU = (MODE & 1) != 0, TAP = (MODE & 2) != 0, CLAMP = (MODE & 4) != 0, RES = (MODE & 8) != 0;
    constexpr int THREADS = TILES * WPT * 32;
    constexpr int ES = I8 ? 1 : 2;                     // bytes of an operand element
    constexpr int UPK = 32 / (8 * ES);                 // units of eight channels per K step
    // Channels transformed at a time on the way in (more shuffles of a stage in flight; four fit the registers of the quantized
    // path: six-layer bf16 chain 380 -> 361 us, unquantized 46.3 -> 46.7) and on the way out (four only pay where the residual's
    // loads are to be covered: 39.8 -> 39.1, chain 361 -> 368).
    constexpr int U = I8 ? 4 : 2, U3 = RES ? 4 : 2;
    // Channels loaded ahead, as one batch: all loads of a batch are issued together and waited for together, a batch later.
    // (Refilled two channels at a time the loads shared scoreboards with younger ones: 39 % of the stalls on bf16.)
    constexpr int NB = (sizeof(T) == 2 && I8) ? 8 : 4;
    constexpr int DQ = (I8 && L == 3) ? 2 : 1;         // dequantization rows per channel
    using TT = HaarTile<L>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_s = tc::smem_u32(smem_raw);
    uint8_t* sm = smem_raw + (((raw_s + 127u) & ~127u) - raw_s);
    const int ksteps = pr.krow / 32;
    const int bpitch = pr.b_resident ? pr.npad : pr.nchunk;                   // rows of the B operand held at a time
    const int bchunks = 2 * (pr.b_resident ? ksteps : pr.ksteps_part);        // 16-byte K chunks of it
    uint8_t* sA = sm;                                                         // [2 * ksteps_part][ROWS][16]
    uint8_t* sB = sA + (size_t)pr.ksteps_part * ROWS * 32;                    // [bchunks][bpitch][16]
    float4* sdq = reinterpret_cast<float4*>(sB + (size_t)bchunks * bpitch * 16);      // I8: [npad][DQ]
    Ctl* ctl = reinterpret_cast<Ctl*>(sdq + (I8 ? pr.npad * DQ : 0));

    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int t = warp & 3, q = warp >> 2;
    // The last, partial wave of tile groups is spread over the SMs that would idle: `parts` CTAs take one group each, all of
    // them build the whole operand and each runs the contraction and the way out for its share of the output channels.
    // (The end of the share costs 25 instantiations a spilled word more than its size would; with the size they took the same time or up
    // to 0.6 % less, but bf16 with three levels and options 1.7 % more: deployed layer of 12 x 64 -> 64 on 96 x 320 59.8 -> 60.9 us.)
    int grp = (int)blockIdx.x, o_lo = 0, o_hi = pr.npad;
    if ((int)blockIdx.x >= pr.split_from) {
        const int r = (int)blockIdx.x - pr.split_from;
        grp = pr.split_from + r / pr.parts;
        o_lo = (r % pr.parts) * pr.share;
        o_hi = min(o_lo + pr.share, pr.npad);
    }
    grp += pr.grp0;
    const bool live = grp * TILES + t < pr.tiles_total;
    const int tiles_x = (pr.W + TT::TW - 1) / TT::TW, tiles_y = pr.H / TT::TH;
    int n, ty, tx;
    tile_coords(min(grp * TILES + t, pr.tiles_total - 1), tiles_x, tiles_y, n, ty, tx);
    const LanePos lp = lane_positions<L>(pr.H, pr.W, ty, tx, lane);
    const size_t P = (size_t)pr.H * pr.W, plane = P * sizeof(T);
    const PatchOff off = patch_off<T>(lp, pr.W);
    const uint64_t xb = reinterpret_cast<uint64_t>(pr.x) + (uint64_t)n * pr.Cin * plane;

    if (WPT == 4) pdl_launch();
    Raw<T> raw[NB];
    const int ureal = (pr.Cin + 7) >> 3;               // units that hold real channels
    auto preload = [&](int u) {
        if (u < ureal) ldg_group<T, VEC, true, true, NB>(xb, plane, off, u * 8, pr.Cin, raw);
    };
    preload(q);

    // ---- set-up -------------------------------------------------------------------------------------
    if (threadIdx.x == 0) {
        tc::mbar_init(tc::smem_u32(&ctl->done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(tc::smem_u32(&ctl->tmem_base)), "r"((uint32_t)pr.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // rows [o0, o0 + rows) of the weights, 16-byte K chunks [j0, j0 + cnt) -> B operand (core-matrix layout)
    auto load_b = [&](int o0, int rows, int j0, int cnt) {
        for (int i = threadIdx.x; i < rows * cnt; i += THREADS) {
            const int row = i / cnt, j = i - row * cnt;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (o0 + row < pr.Cout) v = *reinterpret_cast<const uint4*>(pr.Wq + (size_t)(o0 + row) * pr.krow + (j0 + j) * 16);
            *reinterpret_cast<uint4*>(sB + ((size_t)j * bpitch + row) * 16) = v;
        }
    };
    if (pr.b_resident) load_b(o_lo, o_hi - o_lo, 0, 2 * ksteps);
    // kept or dropped: from the rank map when the select wrote one (thr[n][2] != 0), else by the threshold key
    float nv[8], mul[8];
    int rk[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) nv[s] = (live && slot_ok<L>(lp, s)) ? pr.nrm2[(size_t)n * P + lp.pos[s]] : 0.0f;
    if (WPT == 4 && pr.last) {
        // The launch for the last groups starts when every CTA of the one before it has waited for the selection.  That orders the two in
        // time; what makes the selection's results visible here is the word that the other launch released after its wait.
        // Not seen, although written long ago: wait for that launch as a whole.  Measured against reading on without either: 24 images of
        // 64 -> 64 channels fp32 on 96 x 320 110.5 -> 111.1 us, 12 of them 63.2 -> 63.3.
        uint32_t seen = 1u;
        if (lane == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(pr.selected) : "memory");
        __syncwarp();
        if (__any_sync(0xFFFFFFFFu, seen == 0u)) pdl_wait();
    }
    if (WPT == 2 || !pr.last) pdl_wait();              // what follows reads the selection's results
    // A launch that follows this one for the last groups does not wait for the selection, so it may not run before that is complete.
    if (WPT == 2) {
        if (pr.followed && blockIdx.x == 0 && threadIdx.x == 0)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(pr.selected), "r"(1u) : "memory");
        pdl_launch();
    }
    float amax = 0.0f;
    if (I8) amax = (CLAMP && pr.alpha > 0.0f) ? pr.alpha : *pr.amax_kept;
    {
        const uint4 th = *reinterpret_cast<const uint4*>(pr.thr + n * 4);      // {threshold key, ties kept, use-rank flag, -}
        float inv = 1.0f;
        if (I8) inv = (amax > 0.0f) ? __fdiv_rn(pr.qmax, amax) : 0.0f;
        // the transform runs without its halvings: they go into the per-slot factor (exact, a power of two)
        float sc[8];
        slot_scales<L>(lane, sc);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            rk[s] = -1;
            if (live && slot_ok<L>(lp, s)) {
                if (th.z) rk[s] = pr.rank[(size_t)n * P + lp.pos[s]];
                else rk[s] = (float_key(nv[s]) >= th.x) ? 0 : -1;
            }
            mul[s] = (rk[s] >= 0) ? __fmul_rn(inv, sc[s]) : 0.0f;
        }
    }
    if (I8) {                                          // dequantization factors: scale * 2^-level of every slot pair
        const float scale_a = __fdiv_rn(amax, pr.qmax);
        for (int o = threadIdx.x; o < pr.npad; o += THREADS) {
            const float f = (o < pr.Cout) ? __fmul_rn(scale_a, pr.scale_w[o]) : 0.0f;
            const float s1 = __fmul_rn(f, 0.5f), s2 = __fmul_rn(f, 0.25f);
            if (L == 1) sdq[o] = make_float4(s1, s1, s1, s1);
            else sdq[o * DQ] = make_float4(s1, s1, s2, s2);
            if (L == 3) sdq[o * DQ + DQ - 1] = make_float4(s1, s1, __fmul_rn(f, 0.125f), s2);     // lanes whose slot 6 is of level 3
        }
    }

    const uint32_t a_addr = tc::smem_u32(sA), b_addr = tc::smem_u32(sB), done = tc::smem_u32(&ctl->done);
    const bool clamp = CLAMP && I8 && pr.alpha > 0.0f;         // a given clipping parameter can be exceeded
    const float qmax = pr.qmax;

    // ---- phase 1: transform + quantize the channels of K steps [ks0, ks1) into the A operand ------------------
    auto phase1 = [&](int ks0, int ks1) {
        const int u_end = ks1 * UPK;
        for (int u = ks0 * UPK + q; u < u_end; u += WPT) {
            uint32_t packed[8][2 * ES];                // per slot: 8 int8 codes or 8 bf16 values
            if (u < ureal) {
                Raw<T> cur[NB];
#pragma unroll
                for (int i = 0; i < 8 / U; ++i) {
                    if ((i * U) % NB == 0) {           // the next batch: the other half of this unit, or of the warp's next unit
#pragma unroll
                        for (int d = 0; d < NB; ++d) cur[d] = raw[d];
                        const bool same = NB == 4 && i == 0;
                        const int un = same ? u : u + WPT, c = un * 8 + (same ? 4 : 0);
                        if (un < u_end && un < ureal) {
                            if (c + NB <= pr.Cin) ldg_group<T, VEC, true, false, NB>(xb, plane, off, c, pr.Cin, raw);
                            else ldg_group<T, VEC, true, true, NB>(xb, plane, off, c, pr.Cin, raw);
                        }
                    }
                    float o[U][8];
                    fwd_group<T, L, U>(cur + (i * U) % NB, o, lane);
                    uint32_t code[U][8];
#pragma unroll
                    for (int d = 0; d < U; ++d) {
#pragma unroll
                        for (int s = 0; s < 8; s += 2) {
                            float2 v = mul2(make_float2(o[d][s], o[d][s + 1]), make_float2(mul[s], mul[s + 1]));
                            // int8: the low byte of (v + 1.5*2^23) is the two's complement code of rint(v).  Two scalar
                            // additions of an immediate: a packed addition right after the packed product was contracted
                            // into one fused operation, which changes half-way codes.
                            // clamping before the rounding is the same as after it: the bounds are integers
                            if (CLAMP && clamp) { v.x = fminf(fmaxf(v.x, -qmax), qmax); v.y = fminf(fmaxf(v.y, -qmax), qmax); }
                            code[d][s] = __float_as_uint(I8 ? __fadd_rn(v.x, MAGIC) : v.x);
                            code[d][s + 1] = __float_as_uint(I8 ? __fadd_rn(v.y, MAGIC) : v.y);
                            if (TAP && u * 8 + i * U + d >= pr.Cin) { code[d][s] = 0u; code[d][s + 1] = 0u; }      // the tap's rows are zero padded
                        }
                    }
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        if constexpr (I8) {
                            packed[s][i] = __byte_perm(__byte_perm(code[0][s], code[1][s], 0x0040), __byte_perm(code[2][s], code[3][s], 0x0040), 0x5410);
                        } else {
                            packed[s][i] = pack_bf16x2(__uint_as_float(code[0][s]), __uint_as_float(code[1][s]));
                        }
                    }
                }
            } else {                                   // padding of K up to a whole step
#pragma unroll
                for (int s = 0; s < 8; ++s)
#pragma unroll
                    for (int i = 0; i < 2 * ES; ++i) packed[s][i] = 0u;
            }
            const int ub = (u - ks0 * UPK) * 8 * ES;   // byte offset of the unit inside the part's K range
            uint8_t* dst = sA + ((size_t)(ub >> 4) * ROWS + t * 32 + lane) * 16 + (ub & 15);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                if constexpr (I8) *reinterpret_cast<uint2*>(dst + s * 128 * 16) = make_uint2(packed[s][0], packed[s][1]);
                else *reinterpret_cast<uint4*>(dst + s * 128 * 16) = make_uint4(packed[s][0], packed[s][1], packed[s][2], packed[s][3]);
            }
            if (TAP && pr.xq_tap) {
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    if (rk[s] >= 0) {
                        uint32_t* tp = reinterpret_cast<uint32_t*>(pr.xq_tap + ((size_t)n * pr.k + rk[s]) * pr.krow + (size_t)u * 8 * ES);
#pragma unroll
                        for (int i = 0; i < 2 * ES; ++i) tp[i] = packed[s][i];
                    }
                }
            }
        }
    };

    bool ok = true;
    uint32_t parity = 0;
    const bool k_parts = pr.ksteps_part < ksteps;
    for (int n0 = o_lo; n0 < o_hi && ok; n0 += pr.nchunk) {
        const int cur = min(pr.nchunk, o_hi - n0);
        for (int ks0 = 0; ks0 < ksteps && ok; ks0 += pr.ksteps_part) {
            const int ks1 = min(ksteps, ks0 + pr.ksteps_part);
            if (k_parts && (ks0 > 0 || n0 > o_lo)) preload(ks0 * UPK + q);
            if (k_parts || n0 == o_lo) phase1(ks0, ks1);
            if (!pr.b_resident) load_b(n0, cur, 2 * ks0, 2 * (ks1 - ks0));
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // operands -> visible to the tensor core
            tc::fence_before();
            __syncthreads();
            if (threadIdx.x == 0) {
                tc::fence_after();
                const uint32_t tm = ctl->tmem_base;
                const uint32_t idesc = (I8 ? (2u << 4) : (1u << 4)) | (1u << 7) | (1u << 10) | ((uint32_t)(cur >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
                const int j_b = pr.b_resident ? 2 * ks0 : 0, row_b = pr.b_resident ? n0 - o_lo : 0;
                for (int ks = 0; ks < ks1 - ks0; ++ks) {
                    const uint64_t bd = smem_desc_plain(b_addr + (uint32_t)(((j_b + 2 * ks) * bpitch + row_b) * 16), (uint32_t)bpitch * 16, 128);
#pragma unroll 1
                    for (int b = 0; b < 8; ++b) {
                        const uint64_t ad = smem_desc_plain(a_addr + (uint32_t)((2 * ks * ROWS + b * 128) * 16), ROWS * 16, 128);
                        tc::mma_ss<I8>(tm + (uint32_t)(b * pr.nchunk), ad, bd, idesc, (ks0 + ks) > 0 ? 1u : 0u);
                    }
                }
                tc::mma_commit(done);
            }
            __syncwarp();
            ok = tc::mbar_wait(done, parity);          // the accumulators of this part are complete, the operands may be overwritten
            parity ^= 1u;
            ok = __all_sync(0xFFFFFFFFu, ok ? 1 : 0) != 0;
        }
        tc::fence_after();

        // ---- phase 3: accumulators -> dequantize -> inverse transform -> y ---------------------------------
        const uint32_t taddr = ctl->tmem_base + ((uint32_t)(t * 32) << 16);
        const uint64_t yb = reinterpret_cast<uint64_t>(pr.y) + (uint64_t)n * pr.Cout * plane;
        const uint64_t rb = RES ? reinterpret_cast<uint64_t>(pr.residual) + (uint64_t)n * pr.Cout * plane : 0;
        const bool st0 = live && lp.ok0, st1 = live && lp.ok1;
        const bool coarse6 = L == 3 && ((lane / TT::CG) & 1) == 0;             // slot 6 holds a level-3 coefficient
        const float4* dq = sdq + ((DQ == 2 && coarse6) ? 1 : 0);
        const int groups = min(cur, pr.Cout - n0 + 3) >> 2;                    // groups of four that hold a real channel
        for (int g = q; g < groups && ok; g += WPT) {
            const int o0 = n0 + g * 4;
            uint32_t r[8][4];                          // [slot][channel]
#pragma unroll
            for (int s = 0; s < 8; ++s) tmem_ld4_nowait(taddr + (uint32_t)(s * pr.nchunk + g * 4), r[s]);
            Raw<T> rs[4];
            if (RES && pr.residual) ldg_group<T, VEC, false, true, 4>(rb, plane, off, o0, pr.Cout, rs);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int s = 0; s < 8; ++s) asm volatile("" : "+r"(r[s][0]), "+r"(r[s][1]), "+r"(r[s][2]), "+r"(r[s][3]));
            if (TAP && pr.acc_tap) {
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    if (rk[s] >= 0) {
#pragma unroll
                        for (int d = 0; d < 4; ++d)
                            if (o0 + d < pr.Cout) pr.acc_tap[((size_t)n * pr.k + rk[s]) * pr.Cout + o0 + d] = (int32_t)r[s][d];
                    }
                }
            }
            uint64_t yo = yb + (uint64_t)o0 * plane;
#pragma unroll
            for (int h = 0; h < 4; h += U3) {
                float sl[U3][8], p[U3][2][4];
#pragma unroll
                for (int d = 0; d < U3; ++d) {
                    // dequantize straight into the pre-scaled slots of the inverse: acc * (scale * 2^-level)
                    float4 f;
                    if (I8) f = dq[(o0 + h + d) * DQ];
                    else if (L == 1) f = make_float4(0.5f, 0.5f, 0.5f, 0.5f);
                    else f = make_float4(0.5f, 0.5f, coarse6 ? 0.125f : 0.25f, 0.25f);
#pragma unroll
                    for (int s = 0; s < 8; s += 2) {
                        const float2 a = I8 ? make_float2(__int2float_rn((int)r[s][h + d]), __int2float_rn((int)r[s + 1][h + d]))
                                            : make_float2(__uint_as_float(r[s][h + d]), __uint_as_float(r[s + 1][h + d]));
                        // scalar products: the compiler contracts a packed product with the packed sums of the inverse
                        sl[d][s] = __fmul_rn(a.x, s < 6 ? f.x : f.z);
                        sl[d][s + 1] = __fmul_rn(a.y, s < 6 ? f.y : f.w);
                    }
                }
                inv_group<T, L, U3>(sl, p, lane);
#pragma unroll
                for (int d = 0; d < U3; ++d) {
                    if (RES && pr.residual) {          // y = WCC(x) + residual: one fp32 addition per element (Eq. 13)
#pragma unroll
                        for (int row = 0; row < 2; ++row) {
                            float rp[4];
                            if constexpr (sizeof(T) == 4) {
#pragma unroll
                                for (int i = 0; i < 4; ++i) rp[i] = __uint_as_float(rs[h + d].w[row][i]);
                            } else {
                                rp[0] = bf16lo(rs[h + d].w[row][0]); rp[1] = bf16hi(rs[h + d].w[row][0]);
                                rp[2] = bf16lo(rs[h + d].w[row][1]); rp[3] = bf16hi(rs[h + d].w[row][1]);
                            }
#pragma unroll
                            for (int i = 0; i < 4; ++i) p[d][row][i] = __fadd_rn(p[d][row][i], rp[i]);
                        }
                    }
                    if (RELU && pr.relu) relu_patch(p[d]);
                    if (o0 + h + d < pr.Cout) store_rows<T, VEC>(yo, off, st0, st1, p[d]);
                    yo += plane;
                }
            }
        }
    }

    // ---- tear-down ------------------------------------------------------------------------------------
    if (!ok) {                                         // a wait ran out: report it, give issued work time to finish
        if (lane == 0) atomicExch(pr.status, (int)WCC_ERR_TIMEOUT);
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ctl->tmem_base), "r"((uint32_t)pr.tmem_cols) : "memory");
    }
    if (WPT == 4 && pr.last) pdl_wait();               // complete only after the launch before it: what waits for this one waits for both
}

}  // namespace p2

// Options of the second pass beyond Alg. 1: a given clipping parameter, residual add and ReLU on the way out.
struct FusedExtra { float alpha; int relu; const void* residual; };

// How a layer maps onto the kernel: warps per tile, chunk of output channels in TMEM, K range of the A operand, whether all
// weights stay in shared memory.  Pure arithmetic: callers decide before anything is launched.
struct P2Plan { int wpt, npad, nchunk, ksteps_part, b_resident, tmem_cols; size_t smem; bool ok; };

// Loads in flight live in what the operands leave of an SM's 256 KB to the L1: two CTAs of three K steps each, or one of six,
// leave about 28 KB, and phase 1 then waits on its loads (182 -> 38 channels fp32 on 9 x 176 x 120, second pass alone: 82 us with
// the six steps at once, 53 in two parts).  Two CTAs therefore hold two steps each; see p2_plan for one CTA.
static P2Plan p2_plan_of(int wpt, int Cout, int krow, bool i8, int L, int most_ksteps = 0)
{
    P2Plan p = {};
    p.wpt = wpt;
    p.npad = ceil_div(Cout, 16) * 16;
    const int cap = (wpt == 2) ? 32 : 64;              // 8 slots x cap columns: half of the tensor memory, or all of it
    p.nchunk = p.npad < cap ? p.npad : cap;
    p.tmem_cols = 32;
    while (p.tmem_cols < 8 * p.nchunk) p.tmem_cols <<= 1;
    const int ksteps = krow / 32;
    if (!most_ksteps) most_ksteps = (wpt == 2) ? 2 : ksteps;
    const size_t budget = (wpt == 2) ? 113 * 1024 : 227 * 1024;
    const size_t fixed = 128 + (i8 ? (size_t)p.npad * 16 * (L == 3 ? 2 : 1) : 0) + sizeof(p2::Ctl);
    for (int parts = ceil_div(ksteps, most_ksteps); ; ++parts) {                  // fewest K parts that fit
        p.ksteps_part = ceil_div(ksteps, parts);
        const size_t a = (size_t)p.ksteps_part * p2::ROWS * 32;
        const size_t b_all = (size_t)krow * p.npad, b_chunk = (size_t)p.ksteps_part * 32 * p.nchunk;
        p.b_resident = fixed + a + b_all <= (wpt == 2 ? budget : 195 * 1024);     // (shared memory beyond 196 KB comes out of the L1's last 60)
        p.smem = fixed + a + (p.b_resident ? b_all : b_chunk);
        p.ok = p.smem <= budget;
        if (p.ok || p.ksteps_part == 1) return p;
    }
}

// Two CTAs of eight warps on an SM while there are enough tile groups for it (and the operand does not have to be rebuilt for
// every chunk of output channels): what one CTA waits for, the other covers.  One CTA of sixteen warps otherwise.
// C4 (360 groups) 36.5 against 38.4 us, 24 -> 144 channels on 2 x 256 x 512 (256 groups) 22.8 against 29.5 us; with 128
// groups the sixteen warps win: 96 -> 96 channels on 4 x 128 x 256 23.3 against 32.3 us.  With K in parts of two steps and one
// chunk, two CTAs are 1.0 to 1.4 times as fast from four K steps on (whole layers; 152 -> 10 fp32 on 14 x 76 x 156 52.5 against
// 56.5 us); with two or more chunks and three K steps one CTA is (82 -> 54 fp32 on 2 x 248 x 392 58.6 against 69.4).
// One CTA with one chunk takes K in parts of at most five steps where its loads are what it waits for: six steps in two parts
// from half a wave of groups on (189 -> 45 bf16 on 7 x 296 x 184 159 -> 103 us; below it the second part's first loads cost
// what the L1 gives, +-3 %), more steps from a full wave on (190 -> 42 unquantized fp32 on 6 x 124 x 496 186 -> 148; 247 -> 10
// with 88 groups 37.3 -> 39.2).  Several chunks keep K whole: they would rebuild the operand (192 -> 96 on 4 x 128 x 256 49.7
// against 57.4).
static P2Plan p2_plan(bool two_ctas, int Cout, int krow, bool i8, int L, long long groups, int sms)
{
    const int ksteps = krow / 32;
    const P2Plan two = p2_plan_of(2, Cout, krow, i8, L), one = p2_plan_of(4, Cout, krow, i8, L);
    const bool whole_k = two.ksteps_part == ksteps || two.npad <= two.nchunk;
    if (two_ctas && two.ok && whole_k && groups > sms) return two;
    if (one.npad <= one.nchunk && ksteps > 5 && (ksteps == 6 ? groups * 2 : groups) > sms) return p2_plan_of(4, Cout, krow, i8, L, 5);
    return one;
}

// CTAs that share each of `groups` tile groups by output channels, where they would not fill the SMs otherwise: the split in equal
// parts that one_kernel (libwcc.cu) reckons with, because its lines were measured with it.  Launches use p2_split, which shares more, so
// some layers that are gathered would be faster as one kernel (192 -> 144 bf16 with 36 groups 33.3 gathered, 28.6 as one), but its
// shares alone do not draw the line (256 -> 144 with 24 groups 27.7 and 30.4).
static int p2_shares(long long groups, int sms, int npad)
{
    for (int parts = 4; parts >= 2; parts >>= 1)
        if (groups * parts <= sms && npad % (16 * parts) == 0) return parts;
    return 1;
}

// The split that a launch uses: up to eight CTAs to a group, sixteen channels or more each, the last one perhaps fewer.  Equal parts
// alone (2 or 4, where the padded channels divide) left 3 x 58 -> 70 channels of 60 x 92 bf16, 80 padded channels, to 23 CTAs:
// layer 18.5 us, as 115 CTAs 15.5.  Why as many as there are: of 165 layers with 5 to 72 groups, 1 to 8 K steps and 32 to 256 channels out
// none gained more from fewer than two runs of one split differ (5 %); against equal parts 0.91 of the time (geometric
// mean).  128 -> 256 fp32 with 5 groups, by 1, 2, 4 and 8 CTAs each: 42.2, 30.1, 24.5, 22.1 us; 256 -> 144 bf16 with 24 by 1, 2, 3: 64.1,
// 46.2, 30.7.  Many K steps for few channels out neither gain nor lose (192 -> 64 with 72 groups by 1 and 2: 31.9, 31.7): the SMs that
// build the operand again would idle.
struct P2Split { int parts, share; };
static P2Split p2_split(long long groups, int sms, int npad)
{
    const int units = npad / 16;
    P2Split best = {1, npad};
    for (int parts = 2; parts <= 8 && groups * parts <= sms; ++parts) {
        const int per = ceil_div(units, parts), real = ceil_div(units, per);
        if (real > best.parts) best = {real, per * 16};
    }
    return best;
}

template <typename T, int L, bool VEC>
static wcc_status pass2_dispatch(const void* x, const void* Wq, const int32_t* rank, const float* nrm2, const uint32_t* thr,
                                 const float* amax_kept, int bits, const float* scale_w, int N, int Cin, int Cout, int H, int W,
                                 int k, int kpad, uint32_t* selected, void* y, void* xq_tap, int32_t* acc_tap, const FusedExtra& fx,
                                 cudaStream_t st)
{
    using TT = HaarTile<L>;
    const bool i8 = bits >= 2;
    const int krow = kpad * (i8 ? 1 : 2);
    const long long tiles = (long long)N * ceil_div(W, TT::TW) * (H / TT::TH);
    if (tiles > 0x7FFFFFFFLL) return WCC_ERR_SHAPE;
    const unsigned groups = (unsigned)((tiles + p2::TILES - 1) / p2::TILES);
    DeviceInfo di;
    wcc_status s = device_info(di);
    if (s != WCC_OK) return s;
    const int sms = di.sms;
    const bool tap = xq_tap || acc_tap;
    const P2Plan first = p2_plan(VEC && !tap, Cout, krow, i8, L, groups, sms);
    if (!first.ok) return WCC_ERR_SHAPE;
    p2::Params pr = {};
    pr.x = x; pr.Wq = static_cast<const uint8_t*>(Wq); pr.rank = rank; pr.nrm2 = nrm2; pr.thr = thr; pr.amax_kept = amax_kept;
    pr.scale_w = scale_w; pr.qmax = i8 ? (float)((1 << (bits - 1)) - 1) : 1.0f;
    pr.alpha = fx.alpha; pr.relu = fx.relu; pr.residual = fx.residual;
    pr.N = N; pr.Cin = Cin; pr.Cout = Cout; pr.H = H; pr.W = W; pr.k = k; pr.krow = krow; pr.tiles_total = (int)tiles;
    pr.selected = selected;
    pr.y = y; pr.xq_tap = static_cast<uint8_t*>(xq_tap); pr.acc_tap = acc_tap;
    pr.status = di.status;
    const bool clampv = i8 && fx.alpha > 0.0f;
    const int want = (fx.relu ? 1 : 0) | (tap ? 2 : 0) | (clampv ? 4 : 0) | (fx.residual ? 8 : 0);
    const int mode = want == 0 ? 0 : want == 1 ? 1 : (want & 2) == 0 ? 13 : 15;
    // Groups [g0, g0 + count) by one launch.  The groups of a last, partial wave are shared by output channels when that still fits
    // one wave (the SMs would idle otherwise).
    auto run = [&](const P2Plan& plan, unsigned g0, unsigned count) -> wcc_status {
        pr.npad = plan.npad; pr.nchunk = plan.nchunk; pr.ksteps_part = plan.ksteps_part; pr.b_resident = plan.b_resident;
        pr.tmem_cols = plan.tmem_cols;
        pr.grp0 = (int)g0;
        pr.last = g0 > 0;
        pr.followed = g0 + count < groups;
        const unsigned rem = count % (unsigned)sms;
        const P2Split split = rem > 0 ? p2_split(rem, sms, plan.npad) : P2Split{1, plan.npad};
        pr.parts = split.parts;
        pr.share = split.share;
        pr.split_from = (split.parts > 1) ? (int)(count - rem) : (int)count;
        const unsigned ctas = (unsigned)pr.split_from + (count - (unsigned)pr.split_from) * (unsigned)split.parts;
#define WCC_P2(I8V, WPTV, MODEV)                                                                                     \
        do {                                                                                                        \
            constexpr auto kern = p2::pass2_kernel<T, L, I8V, WPTV, VEC, MODEV>;                                    \
            if ((s = allow_smem<kern>(di.dev, 227 * 1024)) != WCC_OK) return s;                                     \
            return launch_overlapped(kern, dim3(ctas), dim3(p2::TILES * WPTV * 32), plan.smem, st, true, 1, pr);    \
        } while (0)
#define WCC_P2M(I8V, WPTV) do { if (mode == 0) WCC_P2(I8V, WPTV, 0); if (mode == 1) WCC_P2(I8V, WPTV, 1); WCC_P2(I8V, WPTV, 13); } while (0)
        if constexpr (VEC) {
            if (mode != 15) {
                if (i8) { if (plan.wpt == 2) WCC_P2M(true, 2); WCC_P2M(true, 4); }
                if (plan.wpt == 2) WCC_P2M(false, 2);
                WCC_P2M(false, 4);
            }
        } else if (mode == 0) {
            if (i8) WCC_P2(true, 4, 0);
            WCC_P2(false, 4, 0);
        }
        if (i8) WCC_P2(true, 4, 15);
        WCC_P2(false, 4, 15);
#undef WCC_P2M
#undef WCC_P2
    };
    // Two CTAs of eight warps to an SM leave a last wave of up to one CTA per SM at half speed.  Its groups get sixteen warps each, in a
    // launch of their own that takes the SMs as they fall free: 64 -> 64 channels fp32 on 12 x 96 x 320 (360 groups, 64 of them in
    // the last wave) 65.3 -> 63.7 us a layer, 24 images of it (720, 128) 116.0 -> 109.6.  The launch costs up to 2.5 us, so a group must
    // be work enough, of which the way in takes the larger part per channel.  36 layers of 301 to 445 groups, one launch / two: bf16
    // 8 -> 32 channels 25.3 / 27.7, 64 -> 32 50.6 / 50.7, 32 -> 128 46.4 / 46.9, 96 -> 32 49.1 / 48.9, 128 -> 24 58.7 / 56.6, fp32 32 -> 32
    // 36.9 / 37.0, 16 -> 96 49.6 / 48.0, 96 -> 32 72.8 / 68.8.
    const unsigned wave = 2u * (unsigned)sms, last = groups % wave;
    const bool heavy = (int)sizeof(T) * (2 * Cin + Cout) >= 448;
    if (first.wpt == 2 && heavy && groups > wave && last > 0 && last <= (unsigned)sms) {
        const P2Plan rest = p2_plan(false, Cout, krow, i8, L, last, sms);
        if (rest.ok) {
            if ((s = run(first, 0, groups - last)) != WCC_OK) return s;
            return run(rest, groups - last, last);
        }
    }
    return run(first, 0, groups);
}

// Second pass.  xq_tap ([N*k][kpad] of int8 or bf16) and acc_tap (int32 [N*k][Cout]) may be NULL.  *selected is zero.
static wcc_status launch_pass2(const void* x, const void* Wq, const int32_t* rank, const float* nrm2, const uint32_t* thr,
                               const float* amax_kept, int bits, const float* scale_w, int N, int Cin, int Cout, int H, int W,
                               int L, int k, int kpad, wcc_dtype dt, uint32_t* selected, void* y, void* xq_tap, int32_t* acc_tap,
                               const FusedExtra& fx, cudaStream_t st)
{
#define WCC_P2D(TY, LL, VV) return pass2_dispatch<TY, LL, VV>(x, Wq, rank, nrm2, thr, amax_kept, bits, scale_w, N, Cin, Cout, H, W, k, kpad, selected, y, xq_tap, acc_tap, fx, st)
    const bool vec = (W % 4) == 0;                     // always with two or three levels
    if (dt == WCC_F32) {
        if (L == 3) WCC_P2D(float, 3, true);
        if (L == 2) WCC_P2D(float, 2, true);
        if (vec) WCC_P2D(float, 1, true);
        WCC_P2D(float, 1, false);
    }
    if (L == 3) WCC_P2D(__nv_bfloat16, 3, true);
    if (L == 2) WCC_P2D(__nv_bfloat16, 2, true);
    if (vec) WCC_P2D(__nv_bfloat16, 1, true);
    WCC_P2D(__nv_bfloat16, 1, false);
#undef WCC_P2D
}

}  // namespace wcc
