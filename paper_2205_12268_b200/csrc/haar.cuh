// Haar kernels: channel norms of a stored map and the plain inverse (Eq. 3-6, Alg. 1), and the tile geometry all transforms share.
// The forward transform of a feature map is in pass1.cuh, dequantize + scatter + inverse in scatter.cuh.
//
// Work decomposition (all transforms).  One warp owns a tile of 2^L rows x TW columns of one image,
// TW = 4 * CG, CG = 32 / 2^(L-1).  Lane (rp, cg) = (lane / CG, lane % CG) holds the 2 x 4 patch at rows
// 2rp, 2rp+1 and columns 4cg..4cg+3 of the tile: level 1 is computed inside the lane, level 2 pairs the
// lanes rp and rp^1 (lane ^ CG), level 3 combines the four lanes {rp, rp^2} x {cg, cg^1}.  After the
// transform every lane owns exactly eight wavelet-domain positions ("slots"):
//   0,1  y2 of level 1 (two quads)      2,3  y3 of level 1       4,5  y4 of level 1
//   6,7  L=1: y1 of level 1 (two quads)
//        L>=2, rp even: slot 7 = y2 of level 2, slot 6 = y1 of level 2 (L=2) or one of y1..y4 of level 3,
//                       by (rp & 2, cg & 1): (0,0) y1, (0,1) y2, (2,0) y3, (2,1) y4
//        L>=2, rp odd : slot 6 = y3 of level 2, slot 7 = y4 of level 2
// The norm of a position is one chain of fused multiply-adds over the channels in ascending order, whatever warps build it.
// Arithmetic follows the order written in wcc.h so that results are bit-identical to a plain fp32 evaluation.
#pragma once

#include "common.cuh"
#include "tma.cuh"

namespace wcc {

template <int L>
struct HaarTile {
    static constexpr int RP = 1 << (L - 1);   // lane rows
    static constexpr int CG = 32 / RP;        // lane columns
    static constexpr int TH = 2 * RP;         // tile rows  (= 2^L)
    static constexpr int TW = 4 * CG;         // tile columns
};

struct LanePos {
    int pos[8];       // position (row * W + col) of each owned slot inside a plane
    bool ok0, ok1;    // quad 0 / quad 1 of the patch lies inside the image
    int r0, c0;       // top-left of the patch
};

template <int L>
__device__ __forceinline__ LanePos lane_positions(int H, int W, int tile_y, int tile_x, int lane)
{
    using T = HaarTile<L>;
    const int rp = lane / T::CG, cg = lane % T::CG;
    LanePos lp;
    lp.r0 = tile_y * T::TH + 2 * rp;
    lp.c0 = tile_x * T::TW + 4 * cg;
    lp.ok0 = lp.c0 < W;
    lp.ok1 = lp.c0 + 2 < W;
    const int i1 = lp.r0 >> 1, j1 = lp.c0 >> 1, h1 = H >> 1, w1 = W >> 1;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        lp.pos[0 + q] = i1 * W + w1 + j1 + q;
        lp.pos[2 + q] = (h1 + i1) * W + j1 + q;
        lp.pos[4 + q] = (h1 + i1) * W + w1 + j1 + q;
    }
    if (L == 1) {
        lp.pos[6] = i1 * W + j1;
        lp.pos[7] = i1 * W + j1 + 1;
    } else {
        const int i2 = i1 >> 1, j2 = j1 >> 1, h2 = H >> 2, w2 = W >> 2;
        if ((rp & 1) == 0) {
            lp.pos[7] = i2 * W + w2 + j2;
            if (L == 2) {
                lp.pos[6] = i2 * W + j2;
            } else {
                const int i3 = i2 >> 1, j3 = j2 >> 1, h3 = H >> 3, w3 = W >> 3;
                const bool top = (rp & 2) == 0, left = (cg & 1) == 0;
                lp.pos[6] = (top ? i3 : h3 + i3) * W + (left ? j3 : w3 + j3);
            }
        } else {
            lp.pos[6] = (h2 + i2) * W + j2;
            lp.pos[7] = (h2 + i2) * W + w2 + j2;
        }
    }
    return lp;
}

// slot validity: the second quad's level-1 slots (1, 3, 5 and, for L = 1, 7) need ok1
template <int L>
__device__ __forceinline__ bool slot_ok(const LanePos& lp, int s)
{
    if (s < 6) return (s & 1) ? lp.ok1 : lp.ok0;
    if (L == 1) return (s == 7) ? lp.ok1 : lp.ok0;
    return lp.ok0;
}

// Packed fp32 pairs (Blackwell f32x2 pipe): each operation rounds both halves once, to nearest even, exactly like
// the scalar operation.  a - b is written fma(b, -1, a): one rounding of the exact difference.
// add2 / mul2 are written in PTX with an explicit rounding modifier so that a product followed by a sum is never
// contracted into one fused operation (that would round once instead of twice and change quantization codes).
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{\n .reg .b64 ra, rb, rc;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n add.rn.f32x2 rc, ra, rb;\n mov.b64 {%0, %1}, rc;\n}\n"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{\n .reg .b64 ra, rb, rc;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mul.rn.f32x2 rc, ra, rb;\n mov.b64 {%0, %1}, rc;\n}\n"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 half2x(float2 a) { return mul2(a, make_float2(0.5f, 0.5f)); }

// Inverse transform of the lane's eight slots into its patch.
template <int L>
__device__ __forceinline__ void haar_inv_lane(const float (&o)[8], float (&p)[2][4], int lane)
{
    using T = HaarTile<L>;
    float2 ll;
    if (L == 1) {
        ll = make_float2(o[6], o[7]);
    } else {
        const int rp = lane / T::CG, cg = lane % T::CG;
        const float sg = (rp & 1) == 0 ? 1.0f : -1.0f;
        float m0 = o[6];
        if (L == 3) {
            // vertical step: top lanes y1+y3 (y2+y4), bottom lanes y1-y3 (y2-y4); horizontal step: left lanes sum
            // (a, c), right lanes difference (b, d)
            const float sgh = (cg & 1) == 0 ? 1.0f : -1.0f;
            const float sgv = (rp & 2) == 0 ? 1.0f : -1.0f;
            const float pv = __shfl_xor_sync(0xFFFFFFFFu, m0, 2 * T::CG);
            const float w = __fmaf_rn(m0, sgv, pv);
            const float q = __shfl_xor_sync(0xFFFFFFFFu, w, 1);
            const float r = __fmul_rn(__fmaf_rn(w, sgh, q), 0.5f);
            if ((rp & 1) == 0) m0 = r;
        }
        // level 2: upper lane holds (y1, y2), lower lane (y3, y4)
        const float m1 = o[7];
        const float p0 = __shfl_xor_sync(0xFFFFFFFFu, m0, T::CG);
        const float p1 = __shfl_xor_sync(0xFFFFFFFFu, m1, T::CG);
        // upper: (t0, u0) = (y1 + y3, y2 + y4); lower: (t1, u1) = (y1 - y3, y2 - y4)
        const float2 tu = __ffma2_rn(make_float2(m0, m1), make_float2(sg, sg), make_float2(p0, p1));
        ll = make_float2(__fmul_rn(__fadd_rn(tu.x, tu.y), 0.5f), __fmul_rn(__fsub_rn(tu.x, tu.y), 0.5f));
    }
    const float2 y2 = make_float2(o[0], o[1]), y3 = make_float2(o[2], o[3]), y4 = make_float2(o[4], o[5]);
    const float2 t0 = add2(ll, y3), t1 = sub2(ll, y3), u0 = add2(y2, y4), u1 = sub2(y2, y4);
    const float2 a = half2x(add2(t0, u0)), b = half2x(sub2(t0, u0));
    const float2 c = half2x(add2(t1, u1)), d = half2x(sub2(t1, u1));
    p[0][0] = a.x; p[0][1] = b.x; p[0][2] = a.y; p[0][3] = b.y;
    p[1][0] = c.x; p[1][1] = d.x; p[1][2] = c.y; p[1][3] = d.y;
}

// ---- transforms with the halvings taken out ------------------------------------------------------------
// Multiplying by a power of two commutes with every rounding (barring overflow and subnormal results), so the forward
// transform can run on sums and differences alone and leave one exact multiplication per slot to the consumer:
// true coefficient of slot s = raw value * slot_scale[s], where slot_scale = 2^-level.  The same holds for squares
// (norm = raw norm * scale^2) and maxima.  Results are bit-identical to the transform with its halvings while the raw sums of
// squares (up to 4^levels times a norm) stay below 2^128, the raw values below 2^128, and neither squares nor values fall into
// the subnormal range.  Kernels that store coefficients halve at every level and have the whole range.
template <int L>
__device__ __forceinline__ void slot_scales(int lane, float (&sc)[8])
{
    using T = HaarTile<L>;
    const int rp = lane / T::CG;
#pragma unroll
    for (int s = 0; s < 6; ++s) sc[s] = 0.5f;
    if (L == 1) { sc[6] = 0.5f; sc[7] = 0.5f; }
    else {
        sc[7] = 0.25f;
        sc[6] = (L == 3 && (rp & 1) == 0) ? 0.125f : 0.25f;
    }
}

// ---- patch and slot access ------------------------------------------------------------------------
template <typename T, bool VEC>
__device__ __forceinline__ void store_patch(T* __restrict__ plane, int W, const LanePos& lp, const float (&p)[2][4])
{
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        T* dst = plane + (size_t)(lp.r0 + row) * W + lp.c0;
        if (sizeof(T) == 4) {
            if (VEC) {
                if (lp.ok0) *reinterpret_cast<float4*>(dst) = make_float4(p[row][0], p[row][1], p[row][2], p[row][3]);
            } else {
                if (lp.ok0) *reinterpret_cast<float2*>(dst) = make_float2(p[row][0], p[row][1]);
                if (lp.ok1) *reinterpret_cast<float2*>(dst + 2) = make_float2(p[row][2], p[row][3]);
            }
        } else {
            const uint32_t lo = pack_bf16x2(p[row][0], p[row][1]), hi = pack_bf16x2(p[row][2], p[row][3]);
            if (VEC) {
                if (lp.ok0) *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
            } else {
                if (lp.ok0) *reinterpret_cast<uint32_t*>(dst) = lo;
                if (lp.ok1) *reinterpret_cast<uint32_t*>(dst + 2) = hi;
            }
        }
    }
}

// Store the eight slots of a lane into a quadrant-layout fp32 plane.  PAIRS: rows of 4m + 2 store the pairs of the left half, whose
// positions are even, as one (coef_kernel; pass1_kernel is faster without: 12 against 16 us on 293 channels of 4 x 60 x 106 fp32).
template <int L, bool VEC, bool PAIRS = false>
__device__ __forceinline__ void store_slots(float* __restrict__ plane, const LanePos& lp, const float (&o)[8])
{
    if (VEC) {   // W % 4 == 0: both quads valid together and the pairs are 8-byte aligned
        if (lp.ok0) {
            *reinterpret_cast<float2*>(plane + lp.pos[0]) = make_float2(o[0], o[1]);
            *reinterpret_cast<float2*>(plane + lp.pos[2]) = make_float2(o[2], o[3]);
            *reinterpret_cast<float2*>(plane + lp.pos[4]) = make_float2(o[4], o[5]);
            if (L == 1) {
                *reinterpret_cast<float2*>(plane + lp.pos[6]) = make_float2(o[6], o[7]);
            } else {
                plane[lp.pos[6]] = o[6];
                plane[lp.pos[7]] = o[7];
            }
        }
    } else {
#pragma unroll
        for (int s = 0; s < 8; s += 2) {
            if (PAIRS && (s & 2) && lp.ok1) *reinterpret_cast<float2*>(plane + lp.pos[s]) = make_float2(o[s], o[s + 1]);
            else {
                if (slot_ok<L>(lp, s)) plane[lp.pos[s]] = o[s];
                if (slot_ok<L>(lp, s + 1)) plane[lp.pos[s + 1]] = o[s + 1];
            }
        }
    }
}

template <int L, bool VEC>
__device__ __forceinline__ void load_slots(const float* __restrict__ plane, const LanePos& lp, float (&o)[8])
{
    if (VEC) {
        if (lp.ok0) {
            const float2 a = *reinterpret_cast<const float2*>(plane + lp.pos[0]);
            const float2 b = *reinterpret_cast<const float2*>(plane + lp.pos[2]);
            const float2 c = *reinterpret_cast<const float2*>(plane + lp.pos[4]);
            o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y; o[4] = c.x; o[5] = c.y;
            if (L == 1) {
                const float2 d = *reinterpret_cast<const float2*>(plane + lp.pos[6]);
                o[6] = d.x; o[7] = d.y;
            } else {
                o[6] = plane[lp.pos[6]];
                o[7] = plane[lp.pos[7]];
            }
        } else {
#pragma unroll
            for (int s = 0; s < 8; ++s) o[s] = 0.0f;
        }
    } else {
#pragma unroll
        for (int s = 0; s < 8; ++s) o[s] = slot_ok<L>(lp, s) ? plane[lp.pos[s]] : 0.0f;
    }
}

__device__ __forceinline__ void tile_coords(int warp, int tiles_x, int tiles_y, int& n, int& ty, int& tx)
{
    tx = warp % tiles_x;
    const int t = warp / tiles_x;
    ty = t % tiles_y;
    n = t / tiles_y;
}

// Channel norms of a stored coefficient map: one thread per position builds the chain of fused multiply-adds over the
// channels in ascending order, from +0, and max |coef|.  Thirty-two channels of loads in flight per thread.
__global__ void __launch_bounds__(256)
coef_norms_kernel(const float* __restrict__ coef, int N, int C, long long P, float* __restrict__ nrm2, float* __restrict__ amaxpos)
{
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)N * P) return;
    const long long n = id / P, p = id - n * P;
    const float* src = coef + (size_t)n * C * P + p;
    constexpr int UN = 32;
    float acc = 0.0f, am = 0.0f;
    int c = 0;
    for (; c + UN <= C; c += UN) {
        float v[UN];
#pragma unroll
        for (int i = 0; i < UN; ++i) v[i] = __ldcs(src + (size_t)(c + i) * P);
#pragma unroll
        for (int i = 0; i < UN; ++i) {
            acc = __fmaf_rn(v[i], v[i], acc);
            am = fmaxf(am, fabsf(v[i]));
        }
    }
    for (; c < C; ++c) {
        const float v = __ldcs(src + (size_t)c * P);
        acc = __fmaf_rn(v, v, acc);
        am = fmaxf(am, fabsf(v));
    }
    if (nrm2) nrm2[id] = acc;
    if (amaxpos) amaxpos[id] = am;
}

static wcc_status launch_coef_norms(const float* coef, int N, int C, long long P, float* nrm2, float* amaxpos, cudaStream_t st)
{
    if (!nrm2 && !amaxpos) return WCC_OK;
    coef_norms_kernel<<<(unsigned)(((long long)N * P + 255) / 256), 256, 0, st>>>(coef, N, C, P, nrm2, amaxpos);
    WCC_LAUNCH_CHECK();
    return WCC_OK;
}

// ---- plain inverse -------------------------------------------------------------------------------
// One warp per (plane, tile), four or sixteen to a block.
template <typename T, int L, bool VEC>
__global__ void __launch_bounds__(512)
haar_inv_kernel(const float* __restrict__ coef, int planes, int H, int W, T* __restrict__ out)
{
    pdl_wait();
    pdl_launch();
    using TT = HaarTile<L>;
    const int tiles_x = (W + TT::TW - 1) / TT::TW, tiles_y = H / TT::TH;
    const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (warp >= (long long)planes * tiles_x * tiles_y) return;
    const int lane = threadIdx.x & 31;
    int pl, ty, tx;
    tile_coords((int)warp, tiles_x, tiles_y, pl, ty, tx);
    const LanePos lp = lane_positions<L>(H, W, ty, tx, lane);
    const size_t P = (size_t)H * W;
    float o[8], p[2][4];
    load_slots<L, VEC>(coef + (size_t)pl * P, lp, o);
    haar_inv_lane<L>(o, p, lane);
    store_patch<T, VEC>(out + (size_t)pl * P, W, lp, p);
}

// ---- launchers -------------------------------------------------------------------------------
#define WCC_DISPATCH_TLV(FN, dt, L, vec, ...)                                                        \
    do {                                                                                             \
        if ((dt) == WCC_F32) {                                                                       \
            if ((L) == 1) return (vec) ? FN<float, 1, true>(__VA_ARGS__) : FN<float, 1, false>(__VA_ARGS__); \
            if ((L) == 2) return FN<float, 2, true>(__VA_ARGS__);                                    \
            return FN<float, 3, true>(__VA_ARGS__);                                                  \
        } else {                                                                                     \
            if ((L) == 1) return (vec) ? FN<__nv_bfloat16, 1, true>(__VA_ARGS__) : FN<__nv_bfloat16, 1, false>(__VA_ARGS__); \
            if ((L) == 2) return FN<__nv_bfloat16, 2, true>(__VA_ARGS__);                            \
            return FN<__nv_bfloat16, 3, true>(__VA_ARGS__);                                          \
        }                                                                                            \
    } while (0)

template <typename T, int L, bool VEC>
static wcc_status haar_inv_dispatch(const float* coef, int planes, int H, int W, void* out, cudaStream_t st)
{
    using TT = HaarTile<L>;
    const long long warps = (long long)planes * ceil_div(W, TT::TW) * (H / TT::TH);
    // Blocks that wait for the launch before them come and go at one a nanosecond at most.  Four warps move up to 6 or 8 KB, as much
    // as memory does in that time, where the tiles are full; tiles that are not take sixteen warps a block (148 x 14 planes of
    // 346 x 16 bf16 92 -> 66 us; 64 x 180 x 360, full, 3 images of it as blocks of sixteen 62.7 instead of 56.1 for the case).
    const int wpb = (long long)W * (4 + (int)sizeof(T)) * 2 >= 11LL * ceil_div(W, TT::TW) * TT::TW ? 4 : 16;
    const int blocks = (int)((warps + wpb - 1) / wpb);
    return launch_overlapped(haar_inv_kernel<T, L, VEC>, dim3(blocks), dim3(32 * wpb), 0, st, true, 1, coef, planes, H, W, static_cast<T*>(out));
}

wcc_status launch_haar_inv(const float* coef, int N, int C, int H, int W, int L, wcc_dtype dt,
                           void* out, cudaStream_t st)
{
    const bool vec = (W % 4) == 0;
    WCC_DISPATCH_TLV(haar_inv_dispatch, dt, L, vec, coef, N * C, H, W, out, st);
}

}  // namespace wcc
