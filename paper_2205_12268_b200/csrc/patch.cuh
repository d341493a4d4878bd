// A lane's 2 x 4 patch of several channels at once: loads straight from global memory into registers, the forward and the
// inverse transform on them without the halvings of Eq. 3, and stores.  Shared by the kernels of the fused layer.
#pragma once

#include "haar.cuh"

namespace wcc {

// Global accesses as (warp-uniform base, 32-bit lane offset): the form with the fewest address instructions (one 64-bit add
// per access; pointers advanced per lane took 60 % more integer instructions).  NC: read-only data, no L1 allocation.
template <bool NC>
__device__ __forceinline__ void ld_row(uint64_t base, uint32_t off, uint32_t (&w)[4])
{
    if (NC)
        asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %5;\n add.u64 a, a, %4;\n ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [a];\n}\n"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(base), "r"(off));
    else
        asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %5;\n add.u64 a, a, %4;\n ld.global.v4.u32 {%0,%1,%2,%3}, [a];\n}\n"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(base), "r"(off) : "memory");
}
template <bool NC>
__device__ __forceinline__ void ld_row(uint64_t base, uint32_t off, uint32_t (&w)[2])
{
    if (NC)
        asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %3;\n add.u64 a, a, %2;\n ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [a];\n}\n"
                     : "=r"(w[0]), "=r"(w[1]) : "l"(base), "r"(off));
    else
        asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %3;\n add.u64 a, a, %2;\n ld.global.v2.u32 {%0,%1}, [a];\n}\n"
                     : "=r"(w[0]), "=r"(w[1]) : "l"(base), "r"(off) : "memory");
}
__device__ __forceinline__ void st_row(uint64_t base, uint32_t off, float4 v)
{
    asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %1;\n add.u64 a, a, %0;\n st.global.v4.f32 [a], {%2,%3,%4,%5};\n}\n"
                 ::"l"(base), "r"(off), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_row(uint64_t base, uint32_t off, uint2 v)
{
    asm volatile("{\n .reg .u64 a;\n cvt.u64.u32 a, %1;\n add.u64 a, a, %0;\n st.global.v2.u32 [a], {%2,%3};\n}\n"
                 ::"l"(base), "r"(off), "r"(v.x), "r"(v.y) : "memory");
}

// a - b in packed pairs without a constant operand: sub2's fma(b, -1, a) needs the pair (-1, -1), which the compiler rebuilds
// from two moves at every use in a kernel that is short of registers (20 moves per patch in the second pass).
__device__ __forceinline__ float2 diff2(float2 a, float2 b)
{
    float2 r;
    asm("{\n .reg .b64 ra, rb, rc;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n sub.rn.f32x2 rc, ra, rb;\n mov.b64 {%0, %1}, rc;\n}\n"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

template <typename T> struct Raw { uint32_t w[2][sizeof(T)]; };         // two rows of four elements: 4 (fp32) or 2 (bf16) words

// Byte offsets of the lane's two rows inside a plane.  For loads, lanes beyond the right edge (and quads beyond it) are
// redirected to the row's start: what they read is dropped.
struct PatchOff {
    uint32_t o0, o1;          // stores
    uint32_t i0, i1, iq;      // loads: rows, distance of the second quad
};
template <typename T>
__device__ __forceinline__ PatchOff patch_off(const LanePos& lp, int W)
{
    PatchOff f;
    f.o0 = (uint32_t)(((size_t)lp.r0 * W + lp.c0) * sizeof(T));
    f.o1 = f.o0 + (uint32_t)(W * sizeof(T));
    const uint32_t back = (uint32_t)(lp.c0 * sizeof(T));
    f.i0 = lp.ok0 ? f.o0 : f.o0 - back;
    f.i1 = lp.ok0 ? f.o1 : f.o1 - back;
    f.iq = (lp.ok1 ? 2u : 0u) * (uint32_t)sizeof(T);
    return f;
}

// U consecutive channels of the lane's patch starting at channel c; channels beyond the last one repeat it (only a CLIP
// group can have such channels).  `xb`: plane of channel 0.
template <typename T, bool VEC, bool NC, bool CLIP, int U>
__device__ __forceinline__ void ldg_group(uint64_t xb, size_t plane, const PatchOff& f, int c, int C, Raw<T> (&r)[U])
{
    uint64_t b = xb + (uint64_t)(CLIP ? min(c, C - 1) : c) * plane;
#pragma unroll
    for (int d = 0; d < U; ++d) {
#pragma unroll
        for (int row = 0; row < 2; ++row) {
            const uint32_t o = row ? f.i1 : f.i0;
            if constexpr (VEC) {
                ld_row<NC>(b, o, r[d].w[row]);
            } else if constexpr (sizeof(T) == 4) {     // W = 4m + 2 (one level only): the quads are loaded one by one
                uint32_t v[2];
                ld_row<NC>(b, o, v);
                r[d].w[row][0] = v[0]; r[d].w[row][1] = v[1];
                ld_row<NC>(b, o + f.iq, v);
                r[d].w[row][2] = v[0]; r[d].w[row][3] = v[1];
            } else {
                r[d].w[row][0] = *reinterpret_cast<const uint32_t*>(b + o);
                r[d].w[row][1] = *reinterpret_cast<const uint32_t*>(b + o + f.iq);
            }
        }
        if (!CLIP || c + d + 1 < C) b += plane;
    }
}

// Levels 2 and 3 of the forward transform: ll holds the level-1 sums of both quads of the lane, slots 6 and 7 come out.
// HALVE: with the halvings of Eq. 3 (true coefficients); without, sums and differences (see slot_scales).
template <int L, int U, bool HALVE = false>
__device__ __forceinline__ void fwd_levels(const float2 (&ll)[U], float (&o)[U][8], int lane)
{
    using TT = HaarTile<L>;
    if (L == 1) return;
    const int rp = lane / TT::CG, cg = lane % TT::CG;
    const bool even = (rp & 1) == 0;
    const float sg = even ? 1.0f : -1.0f;
    float s[U], dd[U], ps[U], pd[U];
#pragma unroll
    for (int u = 0; u < U; ++u) { s[u] = __fadd_rn(ll[u].x, ll[u].y); dd[u] = __fsub_rn(ll[u].x, ll[u].y); }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        ps[u] = __shfl_xor_sync(0xFFFFFFFFu, s[u], TT::CG);
        pd[u] = __shfl_xor_sync(0xFFFFFFFFu, dd[u], TT::CG);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        o[u][6] = __fmaf_rn(s[u], sg, ps[u]);
        o[u][7] = __fmaf_rn(dd[u], sg, pd[u]);
        if (HALVE) { o[u][6] = __fmul_rn(o[u][6], 0.5f); o[u][7] = __fmul_rn(o[u][7], 0.5f); }
    }
    if (L == 3) {
        const float sgh = (cg & 1) == 0 ? 1.0f : -1.0f;
        const float sgv = (rp & 2) == 0 ? 1.0f : -1.0f;
        float h[U], t[U], q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = __shfl_xor_sync(0xFFFFFFFFu, o[u][6], 1);
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = __fmaf_rn(o[u][6], sgh, h[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = __shfl_xor_sync(0xFFFFFFFFu, t[u], 2 * TT::CG);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float r = __fmaf_rn(t[u], sgv, q[u]);
            if (HALVE) r = __fmul_rn(r, 0.5f);
            if (even) o[u][6] = r;
        }
    }
}

// The first level from the sums and differences of both rows: low-pass values out, slots 0 to 5 (one level: all) written.
template <int L, bool HALVE>
__device__ __forceinline__ void fwd_first(float2 s0, float2 d0, float2 s1, float2 d1, float2& ll, float (&o)[8])
{
    ll = add2(s0, s1);
    float2 y2 = add2(d0, d1), y3 = diff2(s0, s1), y4 = diff2(d0, d1);
    if (HALVE) { ll = half2x(ll); y2 = half2x(y2); y3 = half2x(y3); y4 = half2x(y4); }
    o[0] = y2.x; o[1] = y2.y; o[2] = y3.x; o[3] = y3.y; o[4] = y4.x; o[5] = y4.y;
    if (L == 1) { o[6] = ll.x; o[7] = ll.y; }
}

// Forward transform from the loaded words.  fp32: the first step is scalar,
// because packing (quad 0, quad 1) pairs out of vector loads would take a register move per word (45 instead of 35
// instructions per patch); bf16 words are unpacked anyway, straight into the pairs.
template <typename T, int L, int U, bool HALVE = false>
__device__ __forceinline__ void fwd_group(const Raw<T>* raw, float (&o)[U][8], int lane)
{
    float2 ll[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        float2 s0, d0, s1, d1;
        if constexpr (sizeof(T) == 4) {
            float a[4], c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = __uint_as_float(raw[u].w[0][i]); c[i] = __uint_as_float(raw[u].w[1][i]); }
            s0 = make_float2(__fadd_rn(a[0], a[1]), __fadd_rn(a[2], a[3]));
            d0 = make_float2(__fsub_rn(a[0], a[1]), __fsub_rn(a[2], a[3]));
            s1 = make_float2(__fadd_rn(c[0], c[1]), __fadd_rn(c[2], c[3]));
            d1 = make_float2(__fsub_rn(c[0], c[1]), __fsub_rn(c[2], c[3]));
        } else {
            const float2 a = make_float2(bf16lo(raw[u].w[0][0]), bf16lo(raw[u].w[0][1])), b = make_float2(bf16hi(raw[u].w[0][0]), bf16hi(raw[u].w[0][1]));
            const float2 c = make_float2(bf16lo(raw[u].w[1][0]), bf16lo(raw[u].w[1][1])), d = make_float2(bf16hi(raw[u].w[1][0]), bf16hi(raw[u].w[1][1]));
            s0 = add2(a, b); d0 = diff2(a, b); s1 = add2(c, d); d1 = diff2(c, d);
        }
        fwd_first<L, HALVE>(s0, d0, s1, d1, ll[u], o[u]);
    }
    fwd_levels<L, U, HALVE>(ll, o, lane);
}

// Inverse of slots already multiplied by slot_scales.  fp32: the last step is scalar (the four values of a row leave as one
// vector store).
template <typename T, int L, int U>
__device__ __forceinline__ void inv_group(const float (&o)[U][8], float (&p)[U][2][4], int lane)
{
    using TT = HaarTile<L>;
    float2 ll[U];
    if (L == 1) {
#pragma unroll
        for (int u = 0; u < U; ++u) ll[u] = make_float2(o[u][6], o[u][7]);
    } else {
        const int rp = lane / TT::CG, cg = lane % TT::CG;
        const float sg = (rp & 1) == 0 ? 1.0f : -1.0f;
        float m0[U];
#pragma unroll
        for (int u = 0; u < U; ++u) m0[u] = o[u][6];
        if (L == 3) {
            const float sgh = (cg & 1) == 0 ? 1.0f : -1.0f;
            const float sgv = (rp & 2) == 0 ? 1.0f : -1.0f;
            float pv[U], w[U], q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) pv[u] = __shfl_xor_sync(0xFFFFFFFFu, m0[u], 2 * TT::CG);
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = __fmaf_rn(m0[u], sgv, pv[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = __shfl_xor_sync(0xFFFFFFFFu, w[u], 1);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float r = __fmaf_rn(w[u], sgh, q[u]);
                if ((rp & 1) == 0) m0[u] = r;
            }
        }
        float p0[U], p1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            p0[u] = __shfl_xor_sync(0xFFFFFFFFu, m0[u], TT::CG);
            p1[u] = __shfl_xor_sync(0xFFFFFFFFu, o[u][7], TT::CG);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float tx = __fmaf_rn(m0[u], sg, p0[u]), ty = __fmaf_rn(o[u][7], sg, p1[u]);
            ll[u] = make_float2(__fadd_rn(tx, ty), __fsub_rn(tx, ty));
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const float2 y2 = make_float2(o[u][0], o[u][1]), y3 = make_float2(o[u][2], o[u][3]), y4 = make_float2(o[u][4], o[u][5]);
        const float2 t0 = add2(ll[u], y3), t1 = diff2(ll[u], y3), u0 = add2(y2, y4), u1 = diff2(y2, y4);
        if constexpr (sizeof(T) == 4) {
            p[u][0][0] = __fadd_rn(t0.x, u0.x); p[u][0][1] = __fsub_rn(t0.x, u0.x); p[u][0][2] = __fadd_rn(t0.y, u0.y); p[u][0][3] = __fsub_rn(t0.y, u0.y);
            p[u][1][0] = __fadd_rn(t1.x, u1.x); p[u][1][1] = __fsub_rn(t1.x, u1.x); p[u][1][2] = __fadd_rn(t1.y, u1.y); p[u][1][3] = __fsub_rn(t1.y, u1.y);
        } else {
            const float2 a = add2(t0, u0), b = diff2(t0, u0), c = add2(t1, u1), d = diff2(t1, u1);
            p[u][0][0] = a.x; p[u][0][1] = b.x; p[u][0][2] = a.y; p[u][0][3] = b.y;
            p[u][1][0] = c.x; p[u][1][1] = d.x; p[u][1][2] = c.y; p[u][1][3] = d.y;
        }
    }
}

template <typename T, bool VEC>
__device__ __forceinline__ void store_rows(uint64_t b, const PatchOff& f, bool ok0, bool ok1, const float (&p)[2][4])
{
    if constexpr (VEC) {
        if (ok0) {
#pragma unroll
            for (int row = 0; row < 2; ++row) {
                if constexpr (sizeof(T) == 4) st_row(b, row ? f.o1 : f.o0, make_float4(p[row][0], p[row][1], p[row][2], p[row][3]));
                else st_row(b, row ? f.o1 : f.o0, make_uint2(pack_bf16x2(p[row][0], p[row][1]), pack_bf16x2(p[row][2], p[row][3])));
            }
        }
    } else {
#pragma unroll
        for (int row = 0; row < 2; ++row) {
            const uint64_t dst = b + (row ? f.o1 : f.o0);
            if constexpr (sizeof(T) == 4) {
                if (ok0) *reinterpret_cast<float2*>(dst) = make_float2(p[row][0], p[row][1]);
                if (ok1) *reinterpret_cast<float2*>(dst + 8) = make_float2(p[row][2], p[row][3]);
            } else {
                if (ok0) *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(p[row][0], p[row][1]);
                if (ok1) *reinterpret_cast<uint32_t*>(dst + 4) = pack_bf16x2(p[row][2], p[row][3]);
            }
        }
    }
}

__device__ __forceinline__ void relu_patch(float (&p)[2][4])
{
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = fmaxf(p[a][b], 0.0f);
}

// ---- depthwise 3x3 convolution in front of the transform (stride 1, zero padding 1, cross-correlation) -----------------
// A warp tile with a border of one row and one piece, staged through shared memory by the warp that uses it: a lane needs a
// 4 x 6 neighbourhood of its patch, and out of global memory that was twelve loads with as many 64-bit addresses, their border
// tests or masks on top (202 to 262 instructions per patch); here a lane moves four or five pieces of four elements per
// channel (zeros outside the map) and then reads at constant offsets (181 per patch).  Bound by the shared-memory pipe (70 %
// of its wavefronts) and issue: 1024 channels of 4 x 128 x 128 bf16 convolved, transformed and normed in 96 us.
template <typename T, int L, bool VEC>
struct DwTile {
    using TT = HaarTile<L>;
    static constexpr int ES = (int)sizeof(T);
    static constexpr int PE = VEC ? 4 : 2;             // elements of a piece (rows of 4m + 2 elements: two)
    static constexpr int PW = PE * ES / 4;             // its words
    static constexpr int PR = TT::TW / PE + 2, ROWS = TT::TH + 2, PIECES = PR * ROWS, IT = (PIECES + 31) / 32;
    // bf16, L = 3: two rows of lanes read in one go; this pitch keeps their banks apart
    static constexpr int PITCH = (L == 3 && ES == 2) ? 96 : (TT::TW + 8) * ES;
    static constexpr int CH_BYTES = ROWS * PITCH + 16; // (sixteen bytes take what the last, partial round of pieces writes)
    static constexpr int CHS = 2;                      // channels per stage
    static constexpr int BYTES = 2 * CHS * CH_BYTES;   // two stages

    uint32_t off[IT], dst[IT], valid;
    bool edge;                                         // some piece lies outside the map
    const uint8_t* rd;                                 // this lane's patch in stage 0: row -1, column 0
    uint8_t* wr;

    __device__ __forceinline__ void init(uint8_t* sm, int H, int W, int ty, int tx, int lane)
    {
        valid = 0u;
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int i = lane + 32 * it, row = i / PR, col = i - row * PR;
            const int gr = ty * TT::TH + row - 1, gc = tx * TT::TW + (col - 1) * PE;
            const bool ok = i < PIECES && gr >= 0 && gr < H && gc >= 0 && gc < W;
            off[it] = ok ? (uint32_t)(((long long)gr * W + gc) * ES) : 0u;
            dst[it] = i < PIECES ? (uint32_t)(row * PITCH + (4 + (col - 1) * PE) * ES) : (uint32_t)(ROWS * PITCH);
            valid |= ok ? 1u << it : 0u;
        }
        edge = !__all_sync(0xFFFFFFFFu, valid == (1u << IT) - 1u);
        const int rp = lane / TT::CG, cg = lane % TT::CG;
        rd = sm + 2 * rp * PITCH + (4 + 4 * cg) * ES;
        wr = sm;
    }
    // channels [c, c + CHS), clipped at the last one
    __device__ __forceinline__ void load(uint64_t xb, size_t plane, int c, int C, uint32_t (&w)[CHS][IT][PW]) const
    {
#pragma unroll
        for (int ch = 0; ch < CHS; ++ch) {
            const uint64_t b = xb + (uint64_t)min(c + ch, C - 1) * plane;
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                const uint64_t p = b + off[it];
                if constexpr (PW == 4) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
                    w[ch][it][0] = v.x; w[ch][it][1] = v.y; w[ch][it][2] = v.z; w[ch][it][3] = v.w;
                } else if constexpr (PW == 2) {
                    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
                    w[ch][it][0] = v.x; w[ch][it][1] = v.y;
                } else {
                    w[ch][it][0] = __ldg(reinterpret_cast<const uint32_t*>(p));
                }
            }
        }
    }
    // A __syncwarp has to follow before the stage is read; one between two uses of a stage is enough for its reuse.
    __device__ __forceinline__ void store(int stage, uint32_t (&w)[CHS][IT][PW]) const
    {
        if (edge) {
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                const uint32_t m = ((valid >> it) & 1u) ? 0xFFFFFFFFu : 0u;
#pragma unroll
                for (int ch = 0; ch < CHS; ++ch)
#pragma unroll
                    for (int i = 0; i < PW; ++i) w[ch][it][i] &= m;
            }
        }
        uint8_t* sp = wr + stage * (CHS * CH_BYTES);
#pragma unroll
        for (int ch = 0; ch < CHS; ++ch)
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                uint8_t* d = sp + ch * CH_BYTES + dst[it];
                if constexpr (PW == 4) *reinterpret_cast<uint4*>(d) = make_uint4(w[ch][it][0], w[ch][it][1], w[ch][it][2], w[ch][it][3]);
                else if constexpr (PW == 2) *reinterpret_cast<uint2*>(d) = make_uint2(w[ch][it][0], w[ch][it][1]);
                else *reinterpret_cast<uint32_t*>(d) = w[ch][it][0];
            }
    }
    // The convolution at the eight pixels of the patch, in pairs (columns 0 and 2; 1 and 3), and its first transform level: per
    // pixel one fused multiply-add per tap, row-major tap order, from +0 (taps outside the map meet zeros).  k: taps, duplicated.
    __device__ __forceinline__ void conv(int stage, int ch, const float2* k, float2& ll, float (&o)[8]) const
    {
        const uint8_t* p = rd + stage * (CHS * CH_BYTES) + ch * CH_BYTES;
        float2 e[2], d[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) { e[i] = make_float2(0.0f, 0.0f); d[i] = make_float2(0.0f, 0.0f); }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            float x[6];
            const uint32_t lw = *reinterpret_cast<const uint32_t*>(p + a * PITCH - 4), rw = *reinterpret_cast<const uint32_t*>(p + a * PITCH + 4 * ES);
            if constexpr (ES == 2) {
                const uint2 m = *reinterpret_cast<const uint2*>(p + a * PITCH);
                x[0] = bf16hi(lw);
                x[1] = bf16lo(m.x); x[2] = bf16hi(m.x); x[3] = bf16lo(m.y); x[4] = bf16hi(m.y);
                x[5] = bf16lo(rw);
            } else {
                const float4 m = *reinterpret_cast<const float4*>(p + a * PITCH);
                x[0] = __uint_as_float(lw); x[1] = m.x; x[2] = m.y; x[3] = m.z; x[4] = m.w; x[5] = __uint_as_float(rw);
            }
            const float2 p0 = make_float2(x[0], x[2]), p1 = make_float2(x[1], x[3]), p2 = make_float2(x[2], x[4]), p3 = make_float2(x[3], x[5]);
#pragma unroll
            for (int q = 0; q < 2; ++q) {              // output row q takes tap row a - q
                const int i = a - q;
                if (i < 0 || i > 2) continue;
                e[q] = __ffma2_rn(k[3 * i], p0, e[q]);
                d[q] = __ffma2_rn(k[3 * i], p1, d[q]);
                e[q] = __ffma2_rn(k[3 * i + 1], p1, e[q]);
                d[q] = __ffma2_rn(k[3 * i + 1], p2, d[q]);
                e[q] = __ffma2_rn(k[3 * i + 2], p2, e[q]);
                d[q] = __ffma2_rn(k[3 * i + 2], p3, d[q]);
            }
        }
        fwd_first<L, true>(add2(e[0], d[0]), diff2(e[0], d[0]), add2(e[1], d[1]), diff2(e[1], d[1]), ll, o);
    }
};

// Taps of n consecutive channels from c0 on (n * 9 floats, clipped at the last channel) into shared memory, duplicated, ten
// pairs per channel (80 bytes: rows of sixteen-byte pairs of pairs).
__device__ __forceinline__ void dw_stage_taps(const float* __restrict__ w, int c0, int n, int C, float2* dst, int lane)
{
    for (int e = lane; e < n * 9; e += 32) {
        const int ch = e / 9, t = e - ch * 9;
        const float v = (c0 + ch < C) ? __ldg(w + (size_t)(c0 + ch) * 9 + t) : 0.0f;
        dst[ch * 10 + t] = make_float2(v, v);
    }
}
__device__ __forceinline__ void dw_read_taps(const float2* src, float2 (&k)[10])
{
    const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int i = 0; i < 5; ++i) { const float4 v = s4[i]; k[2 * i] = make_float2(v.x, v.y); k[2 * i + 1] = make_float2(v.z, v.w); }
}

}  // namespace wcc
