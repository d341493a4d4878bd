// Joint shrinkage: per image, the k positions of largest norm (Alg. 1; Eq. 7 with the joint rule).
//
// Radix select on the order-preserving 32-bit key of the fp32 norm, most significant digit first, in three
// rounds of 11 + 11 + 10 bits.  Each round is one kernel: every CTA histograms the digit of the keys of its
// chunk that match the prefix found so far (shared-memory histogram, then one global atomic per non-empty
// bin); the next kernel finds, redundantly in every CTA, the bin that holds the k-th largest key.  After
// the third round the threshold key tau and the number of keys equal to tau that must be kept are known.
// Two more kernels do an ordered stream compaction (chunk counts, then a block scan) so that idx comes out
// ascending and ties go to the lowest position.  Results are deterministic: no output depends on the order
// in which atomics land.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "tma.cuh"

namespace wcc {
namespace cg = cooperative_groups;

constexpr int SEL_THREADS = 256;
constexpr int SEL_KPT = 8;                           // keys per thread
constexpr int SEL_CHUNK = SEL_THREADS * SEL_KPT;     // keys per CTA
constexpr int SEL_BINS = 2048;

// per-image state words
enum { ST_B1 = 0, ST_K1 = 1, ST_B2 = 2, ST_K2 = 3, ST_TAU = 4, ST_NEED_EQ = 5, ST_WORDS = 8 };

struct SelectWs {
    uint32_t* hist;     // [N][3][SEL_BINS]
    float* amax;        // [1] largest |coef| over the kept positions (float bits, merged by integer atomicMax)
    uint32_t* selected; // [1] non-zero once a second pass of two launches has waited for the selection
    uint32_t* bar;      // [N] arrival counters of the per-image barriers of the single-kernel select
    uint32_t* state;    // [N][ST_WORDS]
    uint32_t* chunkcnt; // [N][chunks][2]
    size_t zero_bytes;  // hist + amax + selected + bar are contiguous and cleared together
    int chunks;
};

inline size_t select_ws_bytes(int N, int P)
{
    const size_t chunks = (size_t)ceil_div(P, SEL_CHUNK);
    return align_up((size_t)N * 3 * SEL_BINS * 4, 256) + align_up(64 + (size_t)N * 4, 256) +
           align_up((size_t)N * ST_WORDS * 4, 256) + align_up((size_t)N * chunks * 2 * 4, 256);
}

inline SelectWs carve_select_ws(void* ws, int N, int P)
{
    SelectWs s;
    char* p = static_cast<char*>(ws);
    s.chunks = ceil_div(P, SEL_CHUNK);
    s.hist = reinterpret_cast<uint32_t*>(p);
    p += align_up((size_t)N * 3 * SEL_BINS * 4, 256);
    s.amax = reinterpret_cast<float*>(p);
    s.selected = reinterpret_cast<uint32_t*>(p + 32);
    s.bar = reinterpret_cast<uint32_t*>(p + 64);
    p += align_up(64 + (size_t)N * 4, 256);
    s.zero_bytes = (size_t)(p - static_cast<char*>(ws));
    s.state = reinterpret_cast<uint32_t*>(p);
    p += align_up((size_t)N * ST_WORDS * 4, 256);
    s.chunkcnt = reinterpret_cast<uint32_t*>(p);
    return s;
}

// Block-wide exclusive scan of one value per thread (256 threads); returns the exclusive prefix, total in *total.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_sums, uint32_t* total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += t;
    }
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t s = (lane < SEL_THREADS / 32) ? warp_sums[lane] : 0u;
        uint32_t si = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, si, d);
            if (lane >= d) si += t;
        }
        if (lane < SEL_THREADS / 32) warp_sums[lane] = si - s;     // exclusive warp offsets
        if (lane == SEL_THREADS / 32 - 1) warp_sums[SEL_THREADS / 32] = si;
    }
    __syncthreads();
    const uint32_t res = warp_sums[w] + inc - v;
    *total = warp_sums[SEL_THREADS / 32];
    __syncthreads();
    return res;
}

// Among nbins counts h[] (nbins = 8 * 256 or 4 * 256), find the bin b holding the krem-th key counted from
// the top bin downwards; *above = number of keys in bins > b.  Every thread returns the same values.
template <int NBINS>
__device__ __forceinline__ void find_bin(const uint32_t* __restrict__ h, uint32_t krem, uint32_t* sh_scan,
                                         uint32_t* sh_res, uint32_t& bin, uint32_t& above)
{
    constexpr int PER = NBINS / SEL_THREADS;
    const int top = NBINS - 1 - (int)threadIdx.x * PER;      // this thread covers bins top, top-1, ..., top-PER+1
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) { c[i] = __ldcg(&h[top - i]); sum += c[i]; }
    uint32_t total;
    uint32_t before = block_exclusive_scan(sum, sh_scan, &total);
    if (before < krem && krem <= before + sum) {
        uint32_t a = before;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (a < krem && krem <= a + c[i]) { sh_res[0] = (uint32_t)(top - i); sh_res[1] = a; }
            a += c[i];
        }
    }
    __syncthreads();
    bin = sh_res[0];
    above = sh_res[1];
    __syncthreads();
}

__device__ __forceinline__ void load_keys(const float* __restrict__ v, int P, int base, uint32_t (&key)[SEL_KPT], bool (&ok)[SEL_KPT])
{
    if (base + SEL_KPT <= P && (P % 4) == 0) {
        const float4 a = *reinterpret_cast<const float4*>(v + base);
        const float4 b = *reinterpret_cast<const float4*>(v + base + 4);
        key[0] = float_key(a.x); key[1] = float_key(a.y); key[2] = float_key(a.z); key[3] = float_key(a.w);
        key[4] = float_key(b.x); key[5] = float_key(b.y); key[6] = float_key(b.z); key[7] = float_key(b.w);
#pragma unroll
        for (int i = 0; i < SEL_KPT; ++i) ok[i] = true;
    } else {
#pragma unroll
        for (int i = 0; i < SEL_KPT; ++i) {
            ok[i] = base + i < P;
            key[i] = ok[i] ? float_key(v[base + i]) : 0u;
        }
    }
}

// Round R in {1, 2, 3}: resolve the digit of round R-1 (if any), then histogram digit R of matching keys.
template <int R>
__global__ void __launch_bounds__(SEL_THREADS)
select_hist_kernel(const float* __restrict__ nrm2, int P, int k, uint32_t* __restrict__ hist, uint32_t* __restrict__ state)
{
    __shared__ uint32_t sh[SEL_BINS];
    __shared__ uint32_t sh_scan[SEL_THREADS / 32 + 1];
    __shared__ uint32_t sh_res[2];
    const int n = blockIdx.y;
    uint32_t* hn = hist + (size_t)n * 3 * SEL_BINS;
    uint32_t* stn = state + (size_t)n * ST_WORDS;

    uint32_t prefix = 0;        // digits found so far, right-aligned
    if (R == 2) {
        uint32_t b1, above;
        find_bin<SEL_BINS>(hn, (uint32_t)k, sh_scan, sh_res, b1, above);
        prefix = b1;
        if (blockIdx.x == 0 && threadIdx.x == 0) { stn[ST_B1] = b1; stn[ST_K1] = (uint32_t)k - above; }
    } else if (R == 3) {
        const uint32_t b1 = stn[ST_B1], k1 = stn[ST_K1];
        uint32_t b2, above;
        find_bin<SEL_BINS>(hn + SEL_BINS, k1, sh_scan, sh_res, b2, above);
        prefix = (b1 << 11) | b2;
        if (blockIdx.x == 0 && threadIdx.x == 0) { stn[ST_B2] = b2; stn[ST_K2] = k1 - above; }
    }
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS) sh[i] = 0u;
    __syncthreads();

    uint32_t key[SEL_KPT];
    bool ok[SEL_KPT];
    load_keys(nrm2 + (size_t)n * P, P, blockIdx.x * SEL_CHUNK + threadIdx.x * SEL_KPT, key, ok);
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (R == 1) hist_add(sh, key[i] >> 21, ok[i]);
        if (R == 2) hist_add(sh, (key[i] >> 10) & 0x7FFu, ok[i] && (key[i] >> 21) == prefix);
        if (R == 3) hist_add(sh, key[i] & 0x3FFu, ok[i] && (key[i] >> 10) == prefix);
    }
    __syncthreads();
    uint32_t* out = hn + (R - 1) * SEL_BINS;
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS) {
        const uint32_t c = sh[i];
        if (c) atomicAdd(&out[i], c);
    }
}

// Resolve the last digit; count, per chunk, the keys above and equal to the threshold.
__global__ void __launch_bounds__(SEL_THREADS)
select_count_kernel(const float* __restrict__ nrm2, int P, uint32_t* __restrict__ hist, uint32_t* __restrict__ state,
                    uint32_t* __restrict__ chunkcnt, float* __restrict__ tau)
{
    __shared__ uint32_t sh_scan[SEL_THREADS / 32 + 1];
    __shared__ uint32_t sh_res[2];
    __shared__ uint32_t sh_cnt[2];
    const int n = blockIdx.y;
    uint32_t* hn = hist + (size_t)n * 3 * SEL_BINS;
    uint32_t* stn = state + (size_t)n * ST_WORDS;
    const uint32_t prefix = (stn[ST_B1] << 11) | stn[ST_B2], k2 = stn[ST_K2];
    uint32_t b3, above;
    find_bin<1024>(hn + 2 * SEL_BINS, k2, sh_scan, sh_res, b3, above);
    const uint32_t tkey = (prefix << 10) | b3;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        stn[ST_TAU] = tkey;
        stn[ST_NEED_EQ] = k2 - above;        // how many keys equal to tau are kept (lowest positions first)
        if (tau) tau[n] = key_float(tkey);
    }
    if (threadIdx.x < 2) sh_cnt[threadIdx.x] = 0u;
    __syncthreads();
    uint32_t key[SEL_KPT];
    bool ok[SEL_KPT];
    load_keys(nrm2 + (size_t)n * P, P, blockIdx.x * SEL_CHUNK + threadIdx.x * SEL_KPT, key, ok);
    uint32_t gt = 0, eq = 0;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (!ok[i]) continue;
        gt += key[i] > tkey;
        eq += key[i] == tkey;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        gt += __shfl_xor_sync(0xFFFFFFFFu, gt, d);
        eq += __shfl_xor_sync(0xFFFFFFFFu, eq, d);
    }
    if ((threadIdx.x & 31) == 0) { atomicAdd(&sh_cnt[0], gt); atomicAdd(&sh_cnt[1], eq); }
    __syncthreads();
    if (threadIdx.x < 2) chunkcnt[((size_t)n * gridDim.x + blockIdx.x) * 2 + threadIdx.x] = sh_cnt[threadIdx.x];
}

// Ordered compaction: idx (ascending), rank map, and the largest |coef| over the kept positions.
__global__ void __launch_bounds__(SEL_THREADS)
select_compact_kernel(const float* __restrict__ nrm2, int P, int k, const uint32_t* __restrict__ state,
                      const uint32_t* __restrict__ chunkcnt, int32_t* __restrict__ idx, int32_t* __restrict__ rank,
                      const float* __restrict__ amaxpos, float* __restrict__ amax_kept)
{
    __shared__ uint32_t sh_scan[SEL_THREADS / 32 + 1];
    __shared__ uint32_t sh_base[2];
    __shared__ uint32_t sh_amax;
    const int n = blockIdx.y;
    const uint32_t* stn = state + (size_t)n * ST_WORDS;
    const uint32_t tkey = stn[ST_TAU], need_eq = stn[ST_NEED_EQ];

    // keys above / equal to tau in the chunks before this one
    if (threadIdx.x < 2) sh_base[threadIdx.x] = 0u;
    if (threadIdx.x == 0) sh_amax = 0u;
    __syncthreads();
    {
        uint32_t g = 0, e = 0;
        const uint32_t* cc = chunkcnt + (size_t)n * gridDim.x * 2;
        for (int c = threadIdx.x; c < (int)blockIdx.x; c += SEL_THREADS) { g += cc[2 * c]; e += cc[2 * c + 1]; }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            g += __shfl_xor_sync(0xFFFFFFFFu, g, d);
            e += __shfl_xor_sync(0xFFFFFFFFu, e, d);
        }
        if ((threadIdx.x & 31) == 0 && (g | e)) { atomicAdd(&sh_base[0], g); atomicAdd(&sh_base[1], e); }
    }
    __syncthreads();
    const uint32_t base_gt = sh_base[0], base_eq = sh_base[1];

    uint32_t key[SEL_KPT];
    bool ok[SEL_KPT];
    const int base = blockIdx.x * SEL_CHUNK + threadIdx.x * SEL_KPT;
    load_keys(nrm2 + (size_t)n * P, P, base, key, ok);
    uint32_t gt = 0, eq = 0;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (!ok[i]) continue;
        gt += key[i] > tkey;
        eq += key[i] == tkey;
    }
    uint32_t tot;
    uint32_t gt_before = base_gt + block_exclusive_scan(gt, sh_scan, &tot);
    uint32_t eq_before = base_eq + block_exclusive_scan(eq, sh_scan, &tot);

    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (!ok[i]) continue;
        const bool is_gt = key[i] > tkey, is_eq = key[i] == tkey;
        const bool keep = is_gt || (is_eq && eq_before < need_eq);
        const uint32_t pos = gt_before + min(eq_before, need_eq);
        if (keep) {
            idx[(size_t)n * k + pos] = base + i;
            if (amaxpos) amax = fmaxf(amax, amaxpos[(size_t)n * P + base + i]);
        }
        if (rank) rank[(size_t)n * P + base + i] = keep ? (int32_t)pos : -1;
        gt_before += is_gt;
        eq_before += is_eq;
    }
    if (amax_kept) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
        if ((threadIdx.x & 31) == 0) atomicMax(&sh_amax, __float_as_uint(amax));
        __syncthreads();
        if (threadIdx.x == 0 && sh_amax) atomicMax(reinterpret_cast<uint32_t*>(amax_kept), sh_amax);
    }
}


// ---- the same select as ONE cooperative kernel -------------------------------------------------------
// All phases in one launch; the CTAs of an image meet at per-image barriers (an arrival counter in global memory,
// a bounded spin).  The launch is cooperative, so every CTA is resident and the barriers can complete.  The keys
// stay in registers across the phases.

__device__ __forceinline__ bool image_barrier(uint32_t* counter, uint32_t target)
{
    __shared__ int sh_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(counter, 1u);
        int ok = 0;
        const uint32_t limit = 2u * tc::c_wait_limit;               // polls of >= 40 ns
        for (uint32_t it = 0; it < limit; ++it) {
            if (*reinterpret_cast<volatile uint32_t*>(counter) >= target) { ok = 1; break; }
            __nanosleep(40);
        }
        __threadfence();
        sh_ok = ok;
    }
    __syncthreads();
    return sh_ok != 0;
}

template <int NBINS>
__device__ __forceinline__ void flush_hist(uint32_t* sh, uint32_t* __restrict__ out)
{
    __syncthreads();
    for (int i = threadIdx.x; i < NBINS; i += SEL_THREADS) {
        const uint32_t c = sh[i];
        if (c) atomicAdd(&out[i], c);
        sh[i] = 0u;
    }
}

__global__ void __launch_bounds__(SEL_THREADS)
select_coop_kernel(const float* __restrict__ nrm2, int P, int k, uint32_t* __restrict__ hist, uint32_t* __restrict__ bar,
                   uint32_t* __restrict__ chunkcnt, int32_t* __restrict__ idx, float* __restrict__ tau,
                   int32_t* __restrict__ rank, const float* __restrict__ amaxpos, float* __restrict__ amax_kept,
                   int* __restrict__ status)
{
    __shared__ uint32_t sh[SEL_BINS];
    __shared__ uint32_t sh_scan[SEL_THREADS / 32 + 1];
    __shared__ uint32_t sh_res[2];
    __shared__ uint32_t sh_base[2];
    __shared__ uint32_t sh_amax;
    const int n = blockIdx.y;
    const uint32_t chunks = gridDim.x;
    uint32_t* hn = hist + (size_t)n * 3 * SEL_BINS;
    uint32_t* barn = bar + n;

    uint32_t key[SEL_KPT];
    bool okk[SEL_KPT];
    const int base = blockIdx.x * SEL_CHUNK + threadIdx.x * SEL_KPT;
    load_keys(nrm2 + (size_t)n * P, P, base, key, okk);
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS) sh[i] = 0u;
    if (threadIdx.x < 2) sh_base[threadIdx.x] = 0u;
    if (threadIdx.x == 0) sh_amax = 0u;
    __syncthreads();

    // round 1
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) hist_add(sh, key[i] >> 21, okk[i]);
    flush_hist<SEL_BINS>(sh, hn);
    // A barrier that ran out leaves the histograms incomplete: report it and leave at once (the decision is uniform
    // over the block), so that nothing is derived from them and no index is written.
    auto give_up = [&]() { if (threadIdx.x == 0) atomicExch(status, (int)WCC_ERR_TIMEOUT); };
    if (!image_barrier(barn, chunks)) { give_up(); return; }
    // round 2
    uint32_t b1, above;
    find_bin<SEL_BINS>(hn, (uint32_t)k, sh_scan, sh_res, b1, above);
    const uint32_t k1 = (uint32_t)k - above;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) hist_add(sh, (key[i] >> 10) & 0x7FFu, okk[i] && (key[i] >> 21) == b1);
    flush_hist<SEL_BINS>(sh, hn + SEL_BINS);
    if (!image_barrier(barn, 2 * chunks)) { give_up(); return; }
    // round 3
    uint32_t b2;
    find_bin<SEL_BINS>(hn + SEL_BINS, k1, sh_scan, sh_res, b2, above);
    const uint32_t k2 = k1 - above;
    const uint32_t prefix = (b1 << 11) | b2;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) hist_add(sh, key[i] & 0x3FFu, okk[i] && (key[i] >> 10) == prefix);
    flush_hist<1024>(sh, hn + 2 * SEL_BINS);
    if (!image_barrier(barn, 3 * chunks)) { give_up(); return; }
    // threshold, chunk counts
    uint32_t b3;
    find_bin<1024>(hn + 2 * SEL_BINS, k2, sh_scan, sh_res, b3, above);
    const uint32_t tkey = (prefix << 10) | b3, need_eq = k2 - above;
    if (tau && blockIdx.x == 0 && threadIdx.x == 0) tau[n] = key_float(tkey);
    uint32_t gt = 0, eq = 0;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (!okk[i]) continue;
        gt += key[i] > tkey;
        eq += key[i] == tkey;
    }
    uint32_t tot_gt, tot_eq;
    const uint32_t gt_local = block_exclusive_scan(gt, sh_scan, &tot_gt);
    const uint32_t eq_local = block_exclusive_scan(eq, sh_scan, &tot_eq);
    uint32_t* cc = chunkcnt + (size_t)n * chunks * 2;
    if (threadIdx.x == 0) { cc[2 * blockIdx.x] = tot_gt; cc[2 * blockIdx.x + 1] = tot_eq; }
    if (!image_barrier(barn, 4 * chunks)) { give_up(); return; }
    // ordered compaction
    {
        uint32_t g = 0, e = 0;
        for (int c = threadIdx.x; c < (int)blockIdx.x; c += SEL_THREADS) {
            g += __ldcg(&cc[2 * c]);
            e += __ldcg(&cc[2 * c + 1]);
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            g += __shfl_xor_sync(0xFFFFFFFFu, g, d);
            e += __shfl_xor_sync(0xFFFFFFFFu, e, d);
        }
        if ((threadIdx.x & 31) == 0 && (g | e)) { atomicAdd(&sh_base[0], g); atomicAdd(&sh_base[1], e); }
    }
    __syncthreads();
    uint32_t gt_before = sh_base[0] + gt_local, eq_before = sh_base[1] + eq_local;
    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < SEL_KPT; ++i) {
        if (!okk[i]) continue;
        const bool is_gt = key[i] > tkey, is_eq = key[i] == tkey;
        const bool keep = is_gt || (is_eq && eq_before < need_eq);
        const uint32_t pos = gt_before + min(eq_before, need_eq);
        if (keep && pos < (uint32_t)k) {
            idx[(size_t)n * k + pos] = base + i;
            if (amaxpos) amax = fmaxf(amax, amaxpos[(size_t)n * P + base + i]);
        }
        if (rank) rank[(size_t)n * P + base + i] = keep ? (int32_t)pos : -1;
        gt_before += is_gt;
        eq_before += is_eq;
    }
    if (amax_kept) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
        if ((threadIdx.x & 31) == 0) atomicMax(&sh_amax, __float_as_uint(amax));
        __syncthreads();
        if (threadIdx.x == 0 && sh_amax) atomicMax(reinterpret_cast<uint32_t*>(amax_kept), sh_amax);
    }
}

// ---- the select as one thread-block cluster per image -------------------------------------------------
// Up to 16 CTAs of 256 threads form one cluster per image (P <= 131072 keys, at most 32 per thread, held in registers).  What is
// found in one CTA is pushed into the shared memory of the others (st.shared::cluster, one hardware cluster barrier) instead of
// being read there afterwards; histograms of whole key ranges, needed where the caller supplies none, are combined slice by slice.
// No global-memory round trips between the phases, no spinning, no scratch memory.
constexpr int CL_THREADS = 256;
constexpr int CL_MAXKPT = 32;
constexpr int CL_MAXCS = 16;          // 8 is the portable cluster size; 16 needs the non-portable opt-in
constexpr int CL_CAND_MAX = 2048;    // candidates a CTA has room for (of a gather: CL_CAND_MAX / cs from each CTA); beyond that: another round
constexpr int CL_MSG = 64;           // words of the message in which a CTA sends up to CL_MSG - 1 candidates
constexpr int CL_FEW = 256;          // candidates exchanged by messages
constexpr uint32_t TOO_MANY = 0xFFFFFFFFu, GAVE_UP = 0xFFFFFFFEu;      // instead of a number of candidates (GAVE_UP: or of kept keys)
constexpr int FINE_BINS = 65536;     // histogram of the 16 bits below the sign of every norm, filled by the producer of the norms

struct ClusterSmem {
    union {
        uint32_t hist[SEL_BINS];
        uint32_t local[CL_CAND_MAX];      // this CTA's candidates until they are sent
    };
    uint32_t slice[SEL_BINS];       // sums over all CTAs of this CTA's slice of bins
    uint32_t warp_sums[CL_THREADS / 32 + 1];
    uint32_t warp_gt[CL_THREADS / 32], warp_eq[CL_THREADS / 32];         // (not warp_sums: with a zero threshold no barrier follows its last reading)
    uint32_t slice_total;
    uint32_t res[3];                // found bin, keys above it, keys in it
    uint32_t tot[CL_MAXCS];
    uint32_t amax;
    uint32_t ncand;                 // candidates of this CTA in the gather at hand
    union {
        __align__(16) uint32_t out[1 + CL_CAND_MAX];      // number of this CTA's candidates, candidates; the first CL_MSG words are its message
        uint32_t pushed[CL_CAND_MAX];     // (of a gather) candidates of every CTA of the cluster, CL_CAND_MAX / cs slots each
    };
    __align__(16) uint32_t msg[CL_MAXCS][CL_MSG];  // the messages of all CTAs of the cluster
    uint64_t msg_bar;               // counts their bytes
    __align__(16) uint32_t counts[2][CL_THREADS / 32];         // of a round of rank_by_bits, per warp
    uint32_t pushed_cnt[CL_MAXCS];  // how many each has (more than its slots: none were sent)
    uint2 kept_cnt[CL_MAXCS];       // keys above / equal to the threshold in every CTA; GAVE_UP until it has sent them
    uint32_t narrowing[CL_MAXCS];   // non-zero: the CTA has heard that there are too many candidates for the messages
    __align__(16) uint32_t all[CL_CAND_MAX];      // candidates of all CTAs without gaps
    uint32_t thr[3];                // threshold key, ties to keep, ties in total
    __align__(16) uint32_t range[4];              // positive keys, zeros, smallest positive key, largest key
};

// Store to a CTA of the cluster (addr: this CTA's address of the same variable).
__device__ __forceinline__ void push_u32(uint32_t* addr, int rank, uint32_t v)
{
    asm volatile("{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n st.shared::cluster.u32 [ra], %2;\n}\n" ::"r"(tc::smem_u32(addr)), "r"(rank), "r"(v) : "memory");
}
__device__ __forceinline__ void push_u64(uint2* addr, int rank, uint2 v)
{
    asm volatile("{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n st.shared::cluster.v2.u32 [ra], {%2, %3};\n}\n" ::"r"(tc::smem_u32(addr)), "r"(rank), "r"(v.x), "r"(v.y) : "memory");
}

// Exclusive scan over the threads of a block of CL_THREADS; every thread also gets the total, which warp_sums[WARPS] carries.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t (&warp_sums)[CL_THREADS / 32 + 1], uint32_t* total)
{
    constexpr int WARPS = CL_THREADS / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += t;
    }
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t s = (lane < WARPS) ? warp_sums[lane] : 0u;
        uint32_t si = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, si, d);
            if (lane >= d) si += t;
        }
        if (lane < WARPS) warp_sums[lane] = si - s;
        if (lane == 31) warp_sums[WARPS] = si;
    }
    __syncthreads();
    const uint32_t res = warp_sums[w] + inc - v;
    *total = warp_sums[WARPS];
    __syncthreads();
    return res;
}

// After every CTA has filled sm.hist: find the bin holding the krem-th key from the top over the whole cluster.
// Contains two cluster barriers.  Every thread of every CTA returns the same (bin, above), or false after
// the first barrier if a CTA of the cluster has given up (HIST: see cluster_exchange).
template <bool HIST>
__device__ __forceinline__ bool cluster_find_bin(cg::cluster_group& cluster, ClusterSmem& sm, int cs, int crank, uint32_t krem,
                                                 uint32_t& bin, uint32_t& above)
{
    const int B = SEL_BINS / cs;                     // bins per slice: 128 .. 2048
    cluster.sync();                                  // all local histograms complete
    if (HIST && __any_sync(0xFFFFFFFFu, (int)(threadIdx.x & 31) < cs && sm.narrowing[threadIdx.x & (CL_MAXCS - 1)] == 0u)) return false;
    uint32_t mine = 0;
    for (int t = threadIdx.x; t < B; t += blockDim.x) {
        uint32_t sum = 0;
        for (int r = 0; r < cs; ++r) sum += cluster.map_shared_rank(sm.hist, r)[crank * B + t];
        sm.slice[t] = sum;
        mine += sum;
    }
    uint32_t total;
    block_scan(mine, sm.warp_sums, &total);
    if (threadIdx.x == 0) sm.slice_total = total;
    cluster.sync();                                  // all slices and slice totals complete
    if (threadIdx.x < cs) sm.tot[threadIdx.x] = *cluster.map_shared_rank(&sm.slice_total, threadIdx.x);
    __syncthreads();
    if (threadIdx.x == 0) sm.res[2] = 0u;            // (a barrier follows: the scan's)
    uint32_t above_slices = 0;
    int target = 0;
    bool any = false;                                // (fewer keys than krem: histograms that do not match them)
    for (int r = cs - 1; r >= 0; --r) {              // slices from the top bins downwards
        const uint32_t t = sm.tot[r];
        if (krem <= above_slices + t) { target = r; any = true; break; }
        above_slices += t;
    }
    const uint32_t kin = any ? krem - above_slices : 0u;        // rank inside the target slice, from its top bin
    const uint32_t* rs = cluster.map_shared_rank(sm.slice, target);
    // thread t covers the `per` bins (B-1 - t*per) downwards of the slice (per <= 8)
    const int per = (B + (int)blockDim.x - 1) / (int)blockDim.x;
    const int top = B - 1 - (int)threadIdx.x * per;
    uint32_t c[8], mysum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        c[i] = (i < per && top - i >= 0) ? rs[top - i] : 0u;
        mysum += c[i];
    }
    uint32_t tot2;
    const uint32_t before = block_scan(mysum, sm.warp_sums, &tot2);
    if (before < kin && kin <= before + mysum) {
        uint32_t a = before;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (a < kin && kin <= a + c[i]) { sm.res[0] = (uint32_t)(target * B + top - i); sm.res[1] = above_slices + a; sm.res[2] = c[i]; }
            a += c[i];
        }
    }
    __syncthreads();
    bin = sm.res[0];
    above = sm.res[1];
    __syncthreads();
    return true;
}


// Shift that maps a span of keys onto at most 2048 bins.
__device__ __forceinline__ int span_shift(uint32_t span) { return max(0, 32 - __clz(span) - 11); }

// Gathers the keys in [lo, hi] of the whole cluster into sm.all of every CTA; returns how many there are or TOO_MANY.
// One cluster barrier.  sm.ncand is zero before.
template <int KPT>
__device__ __forceinline__ uint32_t cluster_gather(cg::cluster_group& cluster, ClusterSmem& sm, int cs, int crank, const uint32_t (&key)[KPT], uint32_t in_map,
                                                   uint32_t lo, uint32_t hi, int lane)
{
    uint32_t in = 0u;
#pragma unroll
    for (int i = 0; i < KPT; ++i) in |= (key[i] >= lo && key[i] <= hi) ? 1u << i : 0u;
    in &= in_map;
    if (__any_sync(0xFFFFFFFFu, in != 0u)) {
        uint32_t slot = 0;
        if (in) slot = atomicAdd(&sm.ncand, (uint32_t)__popc(in));
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (in & (1u << i)) {
                if (slot < CL_CAND_MAX) sm.local[slot] = key[i];
                ++slot;
            }
    }
    __syncthreads();
    const uint32_t mine = sm.ncand, slots = CL_CAND_MAX / (uint32_t)cs;
    if ((int)threadIdx.x < cs) push_u32(&sm.pushed_cnt[crank], (int)threadIdx.x, mine);
    if (mine <= slots)
        for (uint32_t t = threadIdx.x; t < mine * (uint32_t)cs; t += blockDim.x)
            push_u32(&sm.pushed[(uint32_t)crank * slots + t / (uint32_t)cs], (int)(t & (uint32_t)(cs - 1)), sm.local[t / (uint32_t)cs]);
    cluster.sync();
    const uint32_t cnt = lane < cs ? sm.pushed_cnt[lane] : 0u, M = __reduce_add_sync(0xFFFFFFFFu, cnt);
    if (__any_sync(0xFFFFFFFFu, cnt > slots)) return TOO_MANY;
    uint32_t upto = cnt;                               // of the CTAs up to `lane`
#pragma unroll
    for (int d = 1; d < CL_MAXCS; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, upto, d);
        if (lane >= d) upto += t;
    }
    for (int r = threadIdx.x >> 5; r < cs; r += CL_THREADS / 32) {
        const uint32_t c = __shfl_sync(0xFFFFFFFFu, cnt, r), at = __shfl_sync(0xFFFFFFFFu, upto, r) - c;
        for (uint32_t j = lane; j < c; j += 32) sm.all[at + j] = sm.pushed[(uint32_t)r * slots + j];
    }
    __syncthreads();
    return M;
}

// Waits for the messages of all CTAs of the cluster, at most so long.
__device__ __forceinline__ bool cluster_listen(ClusterSmem& sm)
{
    const uint32_t bar = tc::smem_u32(&sm.msg_bar), limit = tc::c_wait_limit;
    uint32_t ok = 0;
    for (uint32_t it = 0; it < limit && !ok; ++it)
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0, %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok) : "r"(bar), "r"(1000u) : "memory");
    return ok != 0u;
}

// A CTA whose wait ran out may not leave at once: messages are still on their way to it, and neighbours that heard everything may go
// on to a cluster barrier (histogram rounds, ordered compaction).  It joins one barrier, which ends when every neighbour has left or come
// to its first one, and listens a little longer.  Behind that barrier neighbours look whether all have sent what is sent in
// front of it, and otherwise give up too, without a further barrier.
__device__ __forceinline__ void cluster_give_up(ClusterSmem& sm)
{
    if (threadIdx.x == 0) atomicExch(&g_status, (int)WCC_ERR_TIMEOUT);
    cg::this_cluster().sync();
    cluster_listen(sm);
}

// The short way of a gather: every CTA sends one message of fixed size to every CTA (st.async, counted by the receiver's mbarrier).
// A cluster barrier would also wait for everything that its threads have under way in global memory (its release): 1.6 to 3.4
// us for the gather and its block barriers against 0.8 to 1.3.  Returns how many candidates there are, or GAVE_UP with the status set
// when the wait ran out.  `few`: they are in sm.all.  Otherwise there are more than CL_FEW, or more from a CTA than a message holds.
// st.async is left to launches with the cluster attribute (a lone CTA keeps its candidates): in a launch without it the store faulted
// once, although st.shared::cluster to the own CTA works there.  Nothing documented says why.
template <int KPT>
__device__ __forceinline__ uint32_t cluster_exchange(ClusterSmem& sm, int cs, int crank, const uint32_t (&key)[KPT], uint32_t in_map, uint32_t lo,
                                                     uint32_t hi, int warp, int lane, bool& few)
{
    const bool alone = cs == 1;                        // (a launch without clusters)
    uint32_t in = 0u;
#pragma unroll
    for (int i = 0; i < KPT; ++i) in |= (key[i] >= lo && key[i] <= hi) ? 1u << i : 0u;
    in &= in_map;
    if (__any_sync(0xFFFFFFFFu, in != 0u)) {
        uint32_t* const list = alone ? sm.all : sm.out + 1;
        uint32_t slot = CL_CAND_MAX;
        if (in) slot = atomicAdd(&sm.ncand, (uint32_t)__popc(in));
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (in & (1u << i)) {
                if (slot < CL_CAND_MAX) list[slot] = key[i];
                ++slot;
            }
    }
    __syncthreads();
    if (alone) {
        few = sm.ncand <= CL_FEW;
        return sm.ncand;
    }
    if ((int)threadIdx.x < cs * (CL_MSG / 4)) {        // sixteen bytes to one CTA per thread
        const int to = (int)threadIdx.x / (CL_MSG / 4), j = (int)threadIdx.x % (CL_MSG / 4);
        uint4 w = *reinterpret_cast<const uint4*>(&sm.out[4 * j]);
        if (j == 0) w.x = sm.ncand;
        asm volatile("{\n .reg .b32 ra, rb;\n mapa.shared::cluster.u32 ra, %0, %2;\n mapa.shared::cluster.u32 rb, %1, %2;\n"
                     " st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [ra], {%3, %4, %5, %6}, [rb];\n}\n"
                     ::"r"(tc::smem_u32(&sm.msg[crank][4 * j])), "r"(tc::smem_u32(&sm.msg_bar)), "r"(to), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w) : "memory");
    }
    if (__builtin_expect(!__syncthreads_and(cluster_listen(sm) ? 1 : 0), 0)) {        // (the same for the whole block)
        cluster_give_up(sm);
        return GAVE_UP;
    }
    const uint32_t cnt = lane < cs ? sm.msg[lane][0] : 0u, M = __reduce_add_sync(0xFFFFFFFFu, cnt);
    few = !__any_sync(0xFFFFFFFFu, cnt >= CL_MSG) && M <= CL_FEW;
    if (__builtin_expect(!few, 0)) return M;
    uint32_t upto = cnt;                               // of the CTAs up to `lane`
#pragma unroll
    for (int d = 1; d < CL_MAXCS; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, upto, d);
        if (lane >= d) upto += t;
    }
    for (int r = warp; r < cs; r += CL_THREADS / 32) {
        const uint32_t c = __shfl_sync(0xFFFFFFFFu, cnt, r), at = __shfl_sync(0xFFFFFFFFu, upto, r) - c;
        for (uint32_t j = lane; j < c; j += 32) sm.all[at + j] = sm.msg[r][1 + j];
    }
    __syncthreads();
    return M;
}

// Three bits of the key of rank krem a round, a threshold per warp, until one candidate is left: count(v) and below(v) are the number of
// candidates of v or more and the largest one below v (the same in all lanes of a warp).  All candidates agree with `base` in all but 15 bits.
template <typename Count, typename Below>
__device__ __forceinline__ void rank_by_bits(ClusterSmem& sm, uint32_t M, uint32_t krem, uint32_t base, int warp, int lane, Count count, Below below,
                                             uint32_t& key, uint32_t& need, uint32_t& equal)
{
    uint32_t t = base, above = 0, all = M;             // the key is in [t, t + 2^bits): `all` are t or larger, `above` beyond
    int bits = 15;
#pragma unroll 1
    for (int round = 0; bits > 0 && all - above > 1; ++round) {
        bits -= 3;
        const uint32_t n = count(t + ((uint32_t)warp << bits));
        if (lane == 0) sm.counts[round & 1][warp] = n;
        __syncthreads();
        const uint4 a = *reinterpret_cast<const uint4*>(&sm.counts[round & 1][0]), b = *reinterpret_cast<const uint4*>(&sm.counts[round & 1][4]);
        const uint32_t v[9] = {all, a.y, a.z, a.w, b.x, b.y, b.z, b.w, above};
        uint32_t w = 0;
#pragma unroll
        for (int i = 1; i < 8; ++i)
            if (v[i] >= krem) { w = i; all = v[i]; }
        above = v[8];
#pragma unroll
        for (int i = 7; i >= 1; --i)
            if (v[i] < krem) above = v[i];             // (counts fall with i: ends at the smallest threshold too large)
        t += w << bits;
    }
    if (bits > 0) t = below(t + (1u << bits));         // one candidate left
    key = t; need = krem - above; equal = all - above;
}

// The krem-th largest of the M candidates in sm.all, at most CL_FEW (zeros: none), from registers.
__device__ __forceinline__ void few_rank(ClusterSmem& sm, uint32_t M, uint32_t krem, uint32_t base, int warp, int lane, uint32_t& key, uint32_t& need, uint32_t& equal)
{
    uint32_t c[CL_FEW / 32];
#pragma unroll
    for (int i = 0; i < CL_FEW / 32; ++i) c[i] = sm.all[32 * i + lane];
    auto count = [&](uint32_t v) {
        uint32_t n = 0;
#pragma unroll
        for (int i = 0; i < CL_FEW / 32; ++i) n += c[i] >= v ? 1u : 0u;
        return __reduce_add_sync(0xFFFFFFFFu, n);
    };
    auto below = [&](uint32_t v) {
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < CL_FEW / 32; ++i) m = max(m, c[i] < v ? c[i] : 0u);
        return __reduce_max_sync(0xFFFFFFFFu, m);
    };
    rank_by_bits(sm, M, krem, base, warp, lane, count, below, key, need, equal);
}

// The longer way, for up to CL_CAND_MAX candidates that the messages have counted (M) but could not hold: every CTA writes its own to their
// place in sm.all of every CTA, a warp to one CTA at a time (whole lines; a lane to each took 6 us more for 1920 candidates).  One
// cluster barrier; false behind it if a CTA has given up.  The CTA has sent `narrowing`.  Then as few_rank, from shared memory -> sm.thr.
// Histogram rounds over the cluster instead, as beyond CL_CAND_MAX: one constant map of 64 x 64 14.0 -> 20.7 us a layer, noise in 2 x 64 -> 32
// channels of 256 x 512 bf16, half of it kept, 57.4 -> 61.7.  (Not inlined, so that the short way's code stays together: inlined, six-layer
// chain 324.4 -> 326.7 us, C4 63.5 -> 63.8.)
__device__ __noinline__ bool cluster_spread(ClusterSmem& sm, int cs, int crank, uint32_t M, uint32_t krem, uint32_t base)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < 128 && M + threadIdx.x < CL_CAND_MAX) sm.all[M + threadIdx.x] = 0u;
    if (cs == 1) {                                     // (they are there)
        __syncthreads();
    } else {
        const uint32_t at = __reduce_add_sync(0xFFFFFFFFu, lane < crank ? sm.msg[lane & (CL_MAXCS - 1)][0] : 0u);      // candidates of the CTAs before
        for (int to = warp; to < cs; to += CL_THREADS / 32)
            for (uint32_t j = lane; j < sm.ncand && at + j < CL_CAND_MAX; j += 32) push_u32(&sm.all[at + j], to, sm.out[1 + j]);
        cg::this_cluster().sync();
        if (__any_sync(0xFFFFFFFFu, lane < cs && sm.narrowing[lane & (CL_MAXCS - 1)] == 0u)) return false;
    }
    if (M >= krem) {
        auto count = [&](uint32_t v) {
            uint32_t n = 0;
            for (uint32_t i = 4u * lane; i < M; i += 128) {
                const uint4 x = *reinterpret_cast<const uint4*>(&sm.all[i]);
                n += (x.x >= v) + (x.y >= v) + (x.z >= v) + (x.w >= v);
            }
            return __reduce_add_sync(0xFFFFFFFFu, n);
        };
        auto below = [&](uint32_t v) {
            uint32_t m = 0;
            for (uint32_t i = lane; i < M; i += 32) m = max(m, sm.all[i] < v ? sm.all[i] : 0u);
            return __reduce_max_sync(0xFFFFFFFFu, m);
        };
        uint32_t key, need, equal;
        rank_by_bits(sm, M, krem, base, warp, lane, count, below, key, need, equal);
        if (threadIdx.x == 0) { sm.thr[0] = key; sm.thr[1] = need; sm.thr[2] = equal; }
        __syncthreads();
    }
    return true;
}

// The krem-th largest of the M candidates in sm.all, all of them in [lo, hi] -> sm.thr = {key, equal keys to keep, equal keys}.
// Few are ranked by counting, as many threads to a candidate as there are (one barrier; 168 candidates by one thread each took
// 2.4 us), many by histogram rounds inside the block, eleven bits of the span each (3 us for two rounds, whatever their number).
__device__ __forceinline__ void block_rank(ClusterSmem& sm, uint32_t M, uint32_t krem, uint32_t lo, uint32_t hi)
{
    if (M <= 384) {
        const uint4* all4 = reinterpret_cast<const uint4*>(sm.all);
        uint32_t q = 1;                                // threads per candidate, neighbours in a warp
        while (q < 8 && M * q * 2 <= blockDim.x) q <<= 1;
        const uint32_t part = threadIdx.x & (q - 1);
        for (uint32_t i0 = 0; i0 < M; i0 += blockDim.x / q) {                 // (uniform over the block: whole warps shuffle)
            const uint32_t i = i0 + threadIdx.x / q;
            const uint32_t ci = i < M ? sm.all[i] : 0u;
            uint32_t g = 0, e = 0;
#pragma unroll 4
            for (uint32_t j4 = part; j4 < M / 4; j4 += q) {                   // four candidates per shared-memory load
                const uint4 c = all4[j4];
                g += (c.x > ci) + (c.y > ci) + (c.z > ci) + (c.w > ci);
                e += (c.x == ci) + (c.y == ci) + (c.z == ci) + (c.w == ci);
            }
            if (part == 0)
                for (uint32_t j = M & ~3u; j < M; ++j) { const uint32_t cj = sm.all[j]; g += cj > ci; e += cj == ci; }
            for (uint32_t d = 1; d < q; d <<= 1) {
                g += __shfl_xor_sync(0xFFFFFFFFu, g, d);
                e += __shfl_xor_sync(0xFFFFFFFFu, e, d);
            }
            if (i < M && g < krem && krem <= g + e) { sm.thr[0] = ci; sm.thr[1] = krem - g; sm.thr[2] = e; }      // equal keys write equal values
        }
        __syncthreads();
        return;
    }
    for (;;) {
        const int sh = span_shift(hi - lo);
        for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x) sm.hist[i] = 0u;
        __syncthreads();
        for (uint32_t g = threadIdx.x; g < M; g += blockDim.x) {
            const uint32_t c = sm.all[g];
            if (c >= lo && c <= hi) atomicAdd(&sm.hist[(c - lo) >> sh], 1u);
        }
        __syncthreads();
        constexpr int PER = SEL_BINS / CL_THREADS;
        const int top = SEL_BINS - 1 - (int)threadIdx.x * PER;
        uint32_t c[PER], mysum = 0, tot;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            c[i] = sm.hist[top - i];
            mysum += c[i];
        }
        const uint32_t before = block_scan(mysum, sm.warp_sums, &tot);
        if (before < krem && krem <= before + mysum) {
            uint32_t a = before;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                if (a < krem && krem <= a + c[i]) { sm.res[0] = (uint32_t)(top - i); sm.res[1] = a; sm.res[2] = c[i]; }
                a += c[i];
            }
        }
        __syncthreads();
        const uint32_t b = sm.res[0], above = sm.res[1], cnt = sm.res[2];
        __syncthreads();
        krem -= above;
        lo += b << sh;
        if (sh == 0) {
            if (threadIdx.x == 0) { sm.thr[0] = lo; sm.thr[1] = krem; sm.thr[2] = cnt; }
            __syncthreads();
            return;
        }
        hi = min(hi, lo + ((1u << sh) - 1u));
    }
}

// hist1 ([N][3][2048], round 1 first) and fine ([N][65536]) are optional histograms of the 11 and 16 bits below the sign
// of every norm (norm_digit11 / norm_digit16: norms are never negative) that the producer of the norms filled; with both, the threshold is usually found without any histogram round:
// the 16-bit bin that holds the k-th key contains few keys, which the cluster gathers and ranks directly.
// idx and rank are written only when asked for (want_rank) or when the threshold's ties are kept only in part
// (then the order of positions matters); otherwise consumers compare keys with thr[n] = {threshold key, ties
// kept, use_rank flag, number of candidate keys that were ranked (diagnostic)}.
// A warp owns 32 * KPT consecutive positions, 32 at a time: every load and store is a full line (as consecutive keys per
// thread the loads alone took a microsecond).  The work after the first load is a chain of latencies, so each step is the one
// with the fewest block barriers: warp sums by redux instead of block scans, the owner of the coarse bin goes on to the fine one
// alone, the maxima of what is certainly kept are taken while the cluster barrier is pending.
// Blocks of 256 threads: what every warp has to do besides its keys (some 500 instructions) was most of the issue slots of 1024.
// Measured, from the end of the first pass to the start of the second's threshold (us, blocks of up to 1024 threads that read each
// other's candidates after a cluster barrier -> this): 2 x 131072 positions 14.3 -> 8.3, 12 x 30720 7.8 -> 5.3, 4 x 32768 8.0 -> 6.2.
// KPT: keys per thread (8, 16 or 32; with 32 the 128 registers of two blocks per SM spill 12 bytes, with histograms 32).  HIST: the
// histograms are supplied.  LATE (a test's): the second CTA expects more than is sent to
// it, so its wait runs out.
// False: this CTA has given up, or has not heard from one that has.
template <int KPT, bool HIST, bool LATE>
__device__ __forceinline__ bool cluster_select(ClusterSmem& sm, const float* __restrict__ nrm2, int P, int k, int32_t* __restrict__ idx,
                                               float* __restrict__ tau, int32_t* __restrict__ rank, const float* __restrict__ amaxpos,
                                               float* __restrict__ amax_kept, const uint32_t* __restrict__ hist1, const uint32_t* __restrict__ fine,
                                               uint32_t* __restrict__ thr, int want_rank)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
    const int n = blockIdx.y;
    const float* v = nrm2 + (size_t)n * P;
    constexpr int WARPS = CL_THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = (crank * WARPS + warp) * 32 * KPT + lane;            // this thread's keys: base, base + 32, ...

    if (!HIST)
        for (int i = threadIdx.x; i < SEL_BINS; i += CL_THREADS) sm.hist[i] = 0u;
    if (threadIdx.x < 4) sm.range[threadIdx.x] = threadIdx.x == 2 ? 0xFFFFFFFFu : 0u;
    if (threadIdx.x < CL_MSG) sm.out[threadIdx.x] = 0u;
    for (int i = threadIdx.x; i < CL_FEW; i += CL_THREADS) sm.all[i] = 0u;
    if (HIST && threadIdx.x < CL_MAXCS) { sm.kept_cnt[threadIdx.x].x = GAVE_UP; sm.narrowing[threadIdx.x] = 0u; }
    if (threadIdx.x == 0) {
        tc::mbar_init(tc::smem_u32(&sm.msg_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc::mbar_expect_tx(tc::smem_u32(&sm.msg_bar), (uint32_t)(cs * CL_MSG * 4 + (LATE && crank == 1 ? 16 : 0)));
        sm.amax = 0u;
        sm.ncand = 0u;
        sm.thr[0] = 0xFFFFFFFFu; sm.thr[1] = 0u; sm.thr[2] = 0u;          // keep nothing unless a candidate is found (histograms
        sm.res[0] = 0u; sm.res[1] = 0u; sm.res[2] = 0u;                   // that do not match the keys)
    }
    cluster.barrier_arrive();                          // this CTA runs: others may write to its shared memory
    pdl_wait();
    pdl_launch();
    uint32_t key[KPT], in_map = 0u;                    // in_map: the keys that exist
#pragma unroll
    for (int i = 0; i < KPT; ++i) key[i] = __float_as_uint(__ldcg(v + min(base + 32 * i, P - 1)));      // (no branches: all loads in flight)
    constexpr int PER = SEL_BINS / CL_THREADS;         // coarse bins per thread
    uint4 bins[PER / 4];
    if (HIST) {
        const uint32_t* h = hist1 + (size_t)n * 3 * SEL_BINS + SEL_BINS - 4 - (int)threadIdx.x * PER;
#pragma unroll
        for (int i = 0; i < PER / 4; ++i) bins[i] = __ldcg(reinterpret_cast<const uint4*>(h - 4 * i));
    }
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        key[i] = HIST ? key[i] & 0x7FFFFFFFu : float_key(__uint_as_float(key[i]));       // (norms are never negative)
        in_map |= base + 32 * i < P ? 1u << i : 0u;
    }
    auto valid = [&](int i) { return (in_map & (1u << i)) != 0u; };
    uint32_t am[KPT];                                  // maxima at the positions that may be kept
    auto load_amax = [&](uint32_t limit) {
        const float* a = amaxpos + (size_t)n * P + base;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const uint32_t take = valid(i) && key[i] >= limit ? 1u : 0u;
            asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n mov.u32 %0, 0;\n @p ld.global.cg.u32 %0, [%1];\n}\n" : "=&r"(am[i]) : "l"(a + 32 * i), "r"(take));
        }
    };

    uint32_t tkey = 0, need_eq = 0, total_eq = 0, ranked = 0;    // ranked: candidates counted through (diagnostic)
    uint32_t lo = 0, hi = 0, krem = 0;                 // the threshold is the krem-th largest key in [lo, hi]
    bool found = false, reads_remote = !HIST, amax_loaded = false;
    // The supplied histograms count the non-zero norms only; the zeros are the positions they leave out and rank
    // below everything else.  More kept positions than non-zero norms: the threshold is zero.
    bool zero_thr = false;
    if (HIST) {
        // The 11-bit bin of the threshold: thread t takes the t-th group of bins from the top, the warp that finds the k-th key among
        // its bins goes on to the 16-bit bin (32 fine bins, one per lane, top bin in lane 0).
        uint32_t c[PER], mysum = 0;
#pragma unroll
        for (int i = 0; i < PER; i += 4) {
            const uint4 b = bins[i / 4];
            c[i] = b.w; c[i + 1] = b.z; c[i + 2] = b.y; c[i + 3] = b.x;
            mysum += (b.x + b.y) + (b.z + b.w);
        }
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, mysum);
        if (lane == 0) sm.warp_sums[warp] = wsum;
        __syncthreads();
        const uint32_t ws = lane < WARPS ? sm.warp_sums[lane] : 0u;
        const uint32_t nonzero = __reduce_add_sync(0xFFFFFFFFu, ws), wbefore = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? ws : 0u);
        zero_thr = (uint32_t)k > nonzero;              // the same in every CTA of the cluster
        if (zero_thr) {
            tkey = 0u;                                 // +0
            need_eq = (uint32_t)k - nonzero;
            total_eq = (uint32_t)P - nonzero;
            found = true;
        } else {
            if (wbefore < (uint32_t)k && (uint32_t)k <= wbefore + wsum) {             // one warp
                uint32_t inc = mysum;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                    if (lane >= d) inc += t;
                }
                uint32_t a = wbefore + inc - mysum, b1 = 0, above = 0;
                bool mine = false;
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    if (a < (uint32_t)k && (uint32_t)k <= a + c[i]) { mine = true; b1 = (uint32_t)(SEL_BINS - 1 - (int)threadIdx.x * PER - i); above = a; }
                    a += c[i];
                }
                const int from = __ffs(__ballot_sync(0xFFFFFFFFu, mine)) - 1;
                b1 = __shfl_sync(0xFFFFFFFFu, b1, from);
                const uint32_t k1 = (uint32_t)k - __shfl_sync(0xFFFFFFFFu, above, from);
                const uint32_t bin = (b1 << 5) + 31u - (uint32_t)lane;
                const uint32_t f = __ldcg(&fine[(size_t)n * FINE_BINS + bin]);
                inc = f;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                    if (lane >= d) inc += t;
                }
                const uint32_t before = inc - f;
                if (before < k1 && k1 <= inc) { sm.res[0] = bin; sm.res[1] = k1 - before; }
            }
            __syncthreads();
            lo = max(sm.res[0] << 15, 1u);             // (zeros are not counted)
            hi = lo | 0x7FFFu;
            krem = sm.res[1];
        }
    }
    cluster.barrier_wait();                            // every CTA of the cluster runs
    if (HIST && !found && krem == 0) { tkey = 0xFFFFFFFFu; found = true; }       // no such fine bin: keep nothing, as above
    if (HIST && !found) {
        if (amaxpos) { load_amax(lo); amax_loaded = true; }          // (on their way while the threshold is found)
        bool few;
        const uint32_t M = cluster_exchange<KPT>(sm, cs, crank, key, in_map, lo, hi, warp, lane, few);
        if (__builtin_expect(M == GAVE_UP, 0)) return false;
        if (__builtin_expect(few, 1)) {
            tkey = 0xFFFFFFFFu;                        // keep nothing if there are fewer (histograms that do not match the keys)
            if (M >= krem) few_rank(sm, M, krem, hi & ~0x7FFFu, warp, lane, tkey, need_eq, total_eq);
            ranked = M;
            found = true;
        } else {
            if ((int)threadIdx.x < cs) push_u32(&sm.narrowing[crank], (int)threadIdx.x, 1u);
            if (M <= CL_CAND_MAX) {
                if (!cluster_spread(sm, cs, crank, M, krem, hi & ~0x7FFFu)) return false;
                tkey = sm.thr[0]; need_eq = sm.thr[1]; total_eq = sm.thr[2];
                ranked = M;
                found = true;
            } else {
                reads_remote = true;
                __syncthreads();                       // (a lone CTA has just read its count)
                if (threadIdx.x == 0) sm.ncand = 0u;
                for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x) sm.hist[i] = 0u;
                __syncthreads();
            }
        }
    }
    if (!HIST) {
        // No histograms: the range of the positive keys, and how many keys are positive or zero.  (Zeros would stretch the range
        // by hundreds of octaves; there can be many after a ReLU.)
        uint32_t np = 0, nz = 0, mn = 0xFFFFFFFFu, mx = 0u;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (!valid(i)) continue;
            const bool pos = key[i] > 0x80000000u;
            np += pos;
            nz += key[i] == 0x80000000u;
            mn = min(mn, pos ? key[i] : 0xFFFFFFFFu);
            mx = max(mx, key[i]);
        }
        np = __reduce_add_sync(0xFFFFFFFFu, np);
        nz = __reduce_add_sync(0xFFFFFFFFu, nz);
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (lane == 0) { atomicAdd(&sm.range[0], np); atomicAdd(&sm.range[1], nz); atomicMin(&sm.range[2], mn); atomicMax(&sm.range[3], mx); }
        cluster.sync();
        if (threadIdx.x < 32) {
            uint32_t q[4] = {0u, 0u, 0xFFFFFFFFu, 0u};
            if (lane < cs) {
                const uint4 v = *reinterpret_cast<const uint4*>(cluster.map_shared_rank(sm.range, lane));
                q[0] = v.x; q[1] = v.y; q[2] = v.z; q[3] = v.w;
            }
            q[0] = __reduce_add_sync(0xFFFFFFFFu, q[0]);
            q[1] = __reduce_add_sync(0xFFFFFFFFu, q[1]);
            q[2] = __reduce_min_sync(0xFFFFFFFFu, q[2]);
            q[3] = __reduce_max_sync(0xFFFFFFFFu, q[3]);
            if (lane < 4) sm.tot[lane] = lane == 0 ? q[0] : lane == 1 ? q[1] : lane == 2 ? q[2] : q[3];
        }
        __syncthreads();
        np = sm.tot[0]; nz = sm.tot[1];
        if ((uint32_t)k <= np) { lo = sm.tot[2]; hi = sm.tot[3]; krem = (uint32_t)k; }
        else if ((uint32_t)k <= np + nz) { tkey = 0x80000000u; need_eq = (uint32_t)k - np; total_eq = nz; found = true; }
        else { lo = 0u; hi = 0x7FFFFFFFu; krem = (uint32_t)k - np - nz; }
        __syncthreads();
    }
    // Narrow [lo, hi] until its keys fit the gather: 2048 bins a round over the keys' own range.  For norms (10 to 20 octaves,
    // most keys within two) the first round leaves tens to hundreds of keys; fixed leading digits left thousands, and most
    // counts went to a few bins.
    for (bool first = true; !found; first = false) {
        const int sh = span_shift(hi - lo);
        if (!first) {                                  // (all neighbours have read this CTA's bins)
            if (threadIdx.x == 0) sm.ncand = 0u;
            for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x) sm.hist[i] = 0u;
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const bool in = valid(i) && key[i] >= lo && key[i] <= hi;
            const uint32_t b = (key[i] - lo) >> sh;
            if (in) atomicAdd(&sm.hist[b], 1u);
        }
        uint32_t b, above;
        if (!cluster_find_bin<HIST>(cluster, sm, cs, crank, krem, b, above)) return false;
        const uint32_t cnt = sm.res[2];
        if (HIST && cnt == 0) { tkey = 0xFFFFFFFFu; need_eq = total_eq = 0u; break; }    // fewer keys than the histograms say: keep nothing
        krem -= above;
        lo += b << sh;
        if (sh == 0) { tkey = lo; need_eq = krem; total_eq = cnt; break; }
        hi = min(hi, lo + ((1u << sh) - 1u));
        if (cnt <= CL_CAND_MAX) {
            const uint32_t M = cluster_gather<KPT>(cluster, sm, cs, crank, key, in_map, lo, hi, lane);
            if (M != TOO_MANY) {
                block_rank(sm, M, krem, lo, hi);
                tkey = sm.thr[0]; need_eq = sm.thr[1]; total_eq = sm.thr[2];
                ranked = M;
                break;
            }
        }
    }
    const uint32_t tkey_out = HIST ? tkey | 0x80000000u : tkey;               // as float_key
    if (tau && crank == 0 && threadIdx.x == 0) tau[n] = key_float(tkey_out);

    // Ties kept in part need the order of positions, except ties at zero: a position whose norm is zero holds only zero
    // coefficients, so keeping more of them than asked changes nothing downstream (consumers that get the threshold
    // alone keep every position with key >= threshold).
    const bool split_ties = need_eq < total_eq && !zero_thr;
    const bool ordered = want_rank || split_ties;      // uniform over the cluster
    if (thr && crank == 0 && threadIdx.x == 0) {
        thr[n * 4 + 0] = tkey_out;
        thr[n * 4 + 1] = need_eq;
        thr[n * 4 + 2] = ordered ? 1u : 0u;
        thr[n * 4 + 3] = ranked;
    }
    if (amaxpos && !amax_loaded) load_amax(tkey);
    uint32_t amax = 0u;                                // (bits of a non-negative float: ordered like an integer)
    if (!ordered) {
        // every key >= threshold is kept; nobody needs the order
        if (amaxpos) {
#pragma unroll
            for (int i = 0; i < KPT; ++i)
                if (key[i] >= tkey) amax = max(amax, am[i]);           // (what does not exist has no maximum)
        }
    } else {
        // ordered compaction: ascending idx, rank map, ties to the lowest positions
        uint32_t gt = 0, eq = 0;                       // of the warp
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            gt += (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, valid(i) && key[i] > tkey));
            eq += (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, valid(i) && key[i] == tkey));
        }
        if (lane == 0) { sm.warp_gt[warp] = gt; sm.warp_eq[warp] = eq; }
        __syncthreads();
        const uint32_t wg = lane < WARPS ? sm.warp_gt[lane] : 0u, we = lane < WARPS ? sm.warp_eq[lane] : 0u;
        uint32_t gt_before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wg : 0u), eq_before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? we : 0u);
        const uint32_t tot_gt = __reduce_add_sync(0xFFFFFFFFu, wg), tot_eq = __reduce_add_sync(0xFFFFFFFFu, we);
        if ((int)threadIdx.x < cs) push_u64(&sm.kept_cnt[crank], (int)threadIdx.x, make_uint2(tot_gt, tot_eq));
        cluster.sync();
        const uint2 sent = lane < cs ? sm.kept_cnt[lane] : make_uint2(0u, 0u);
        if (HIST && __any_sync(0xFFFFFFFFu, sent.x == GAVE_UP)) return false;
        gt_before += __reduce_add_sync(0xFFFFFFFFu, lane < crank ? sent.x : 0u);
        eq_before += __reduce_add_sync(0xFFFFFFFFu, lane < crank ? sent.y : 0u);
        const unsigned below = (1u << lane) - 1u;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const bool is_gt = valid(i) && key[i] > tkey, is_eq = valid(i) && key[i] == tkey;
            const unsigned mg = __ballot_sync(0xFFFFFFFFu, is_gt), me = __ballot_sync(0xFFFFFFFFu, is_eq);
            const uint32_t g = gt_before + (uint32_t)__popc(mg & below), e = eq_before + (uint32_t)__popc(me & below);
            const uint32_t pos = g + min(e, need_eq);
            const bool keep = (is_gt || (is_eq && e < need_eq)) && pos < (uint32_t)k;          // (beyond k: only where the histograms do not match)
            if (keep) {
                if (idx) idx[(size_t)n * k + pos] = base + 32 * i;
                if (amaxpos) amax = max(amax, am[i]);
            }
            if (rank && valid(i)) rank[(size_t)n * P + base + 32 * i] = keep ? (int32_t)pos : -1;
            gt_before += (uint32_t)__popc(mg);
            eq_before += (uint32_t)__popc(me);
        }
    }
    if (amax_kept) {
        amax = __reduce_max_sync(0xFFFFFFFFu, amax);
        if (lane == 0 && amax) atomicMax(&sm.amax, amax);
        __syncthreads();
        if (threadIdx.x == 0 && sm.amax) atomicMax(reinterpret_cast<uint32_t*>(amax_kept), sm.amax);
    }
    if (reads_remote) cluster.sync();                  // nobody leaves while a neighbour may still read its shared memory
    return true;
}

template <int KPT, bool HIST, bool LATE = false>
__global__ void __launch_bounds__(CL_THREADS, 2)
select_cluster_kernel(const float* __restrict__ nrm2, int P, int k, int32_t* __restrict__ idx, float* __restrict__ tau,
                      int32_t* __restrict__ rank, const float* __restrict__ amaxpos, float* __restrict__ amax_kept,
                      const uint32_t* __restrict__ hist1, const uint32_t* __restrict__ fine, uint32_t* __restrict__ thr,
                      int want_rank)
{
    __shared__ ClusterSmem sm;
    if (cluster_select<KPT, HIST, LATE>(sm, nrm2, P, k, idx, tau, rank, amaxpos, amax_kept, hist1, fine, thr, want_rank)) return;
    // none of this CTA's positions is kept
    const int from = (int)blockIdx.x * CL_THREADS * KPT, n = blockIdx.y;
    if (rank)
        for (int p = from + (int)threadIdx.x; p < min(from + CL_THREADS * KPT, P); p += CL_THREADS) rank[(size_t)n * P + p] = -1;
    if (thr && blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<uint4*>(thr + n * 4) = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
}

__global__ void thr_use_rank_kernel(uint32_t* thr, int N)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n < N) { thr[n * 4 + 0] = 0u; thr[n * 4 + 1] = 0u; thr[n * 4 + 2] = 1u; }
}

// One cluster per image holds up to this many positions in registers (the path that uses a producer's histograms).
inline bool select_in_cluster(int P) { return P <= CL_MAXCS * CL_THREADS * CL_MAXKPT; }

// hist1_ready: the caller has already cleared the zero region of the workspace (carve_select_ws(...).hist,
// zero_bytes) and filled round 1 of the histogram (norm_digit11 of every non-zero norm) before this call.
// fine / thr: see select_cluster_kernel; want_rank: idx (if non-NULL) and rank must be written even when the
// threshold alone would do.  Without thr the rank map and idx are always written.
wcc_status launch_select(const float* nrm2, int N, int P, int k, int32_t* idx, float* tau,
                         int32_t* rank, const float* amaxpos, bool want_amax,
                         void* ws, size_t ws_bytes, cudaStream_t st, bool hist1_ready,
                         const uint32_t* fine, uint32_t* thr, bool want_rank)
{
    if (ws_bytes < select_ws_bytes(N, P)) return WCC_ERR_WORKSPACE;
    const SelectWs s = carve_select_ws(ws, N, P);
    float* amax_kept = want_amax ? s.amax : nullptr;
    // one cluster per image while its keys fit in the registers of 16 x 256 threads, when the device schedules clusters of 16 CTAs (opt-in)
    static std::atomic<int> max_cs[MAX_DEVICES];       // 0: not asked yet (threads that ask at the same time find the same)
    int devc = 0;
    WCC_CUDA_TRY(cudaGetDevice(&devc));
    const bool known = devc >= 0 && devc < MAX_DEVICES;
    int cs_cap = known ? max_cs[devc].load(std::memory_order_relaxed) : 8;
    if (cs_cap == 0) {
        cs_cap = 8;
        bool all = true;
        auto allow16 = [&](auto kern) { all = all && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess; };
        allow16(select_cluster_kernel<8, true>); allow16(select_cluster_kernel<16, true>); allow16(select_cluster_kernel<CL_MAXKPT, true>);
        allow16(select_cluster_kernel<8, false>); allow16(select_cluster_kernel<16, false>); allow16(select_cluster_kernel<CL_MAXKPT, false>);
        if (all) {
            cudaLaunchConfig_t q = {};
            q.gridDim = dim3(16, 1);
            q.blockDim = dim3(CL_THREADS);
            cudaLaunchAttribute qa[1];
            qa[0].id = cudaLaunchAttributeClusterDimension;
            qa[0].val.clusterDim.x = 16; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
            q.attrs = qa; q.numAttrs = 1;
            int nclusters = 0;
            if (cudaOccupancyMaxActiveClusters(&nclusters, select_cluster_kernel<CL_MAXKPT, true>, &q) == cudaSuccess && nclusters > 0) cs_cap = 16;
        }
        (void)cudaGetLastError();
        max_cs[devc].store(cs_cap, std::memory_order_relaxed);
    }
    if (select_in_cluster(P) && P <= cs_cap * CL_THREADS * CL_MAXKPT) {
        int cs = 1;
        while (cs < cs_cap && cs * CL_THREADS * 8 < P) cs <<= 1;        // about eight keys per thread,
        while (cs > 1 && (long long)N * cs > 2 * B200_SMS && P <= cs / 2 * CL_THREADS * CL_MAXKPT) cs >>= 1;      // all images in one wave
        const int kpt = ceil_div(P, cs * CL_THREADS);
        if (amax_kept && !hist1_ready) WCC_CUDA_TRY(cudaMemsetAsync(amax_kept, 0, sizeof(float), st));
        const uint32_t* hist1 = hist1_ready ? s.hist : nullptr;
        const uint32_t* fine_use = hist1_ready ? fine : (const uint32_t*)nullptr;
        const int wr = (want_rank || !thr) ? 1 : 0;
        auto go = [&](auto kern) -> wcc_status {
            return launch_overlapped(kern, dim3(cs, N), dim3(CL_THREADS), 0, st, true, cs, nrm2, P, k, idx, tau, rank, amaxpos, amax_kept,
                                     hist1, fine_use, thr, wr);
        };
        // few keys per thread: the instantiations with fewer key registers
        if (hist1_ready && fine)
            return kpt <= 8 ? go(select_cluster_kernel<8, true>) : kpt <= 16 ? go(select_cluster_kernel<16, true>) : go(select_cluster_kernel<CL_MAXKPT, true>);
        return kpt <= 8 ? go(select_cluster_kernel<8, false>) : kpt <= 16 ? go(select_cluster_kernel<16, false>) : go(select_cluster_kernel<CL_MAXKPT, false>);
    }
    if (thr) {                                        // these paths always write idx and the rank map
        thr_use_rank_kernel<<<ceil_div(N, 128), 128, 0, st>>>(thr, N);
        ++g_launches;
    }
    // (histograms supplied by the caller are not used by these paths: they start from a clean slate)
    WCC_CUDA_TRY(cudaMemsetAsync(s.hist, 0, s.zero_bytes, st));
    const dim3 grid(s.chunks, N);

    // one cooperative kernel when every CTA can be resident at once, else one kernel per phase
    static int coop_cap[64] = {0};          // per device: 0 unknown, -1 unsupported, else max resident CTAs
    int dev = 0;
    WCC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && coop_cap[dev] == 0) {
        int coop = 0, sms = 0, per_sm = 0;
        WCC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        WCC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        WCC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, select_coop_kernel, SEL_THREADS, 0));
        coop_cap[dev] = (coop && per_sm > 0) ? sms * per_sm : -1;
    }
    const long long ctas = (long long)s.chunks * N;
    if (dev >= 0 && dev < 64 && coop_cap[dev] > 0 && ctas <= coop_cap[dev]) {
        int* status = nullptr;
        WCC_CUDA_TRY(cudaGetSymbolAddress(reinterpret_cast<void**>(&status), g_status));
        uint32_t* hist = s.hist; uint32_t* bar = s.bar; uint32_t* chunkcnt = s.chunkcnt;
        void* args[] = {(void*)&nrm2, (void*)&P, (void*)&k, (void*)&hist, (void*)&bar, (void*)&chunkcnt, (void*)&idx,
                        (void*)&tau, (void*)&rank, (void*)&amaxpos, (void*)&amax_kept, (void*)&status};
        WCC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(select_coop_kernel), grid, dim3(SEL_THREADS), args, 0, st));
        WCC_LAUNCH_CHECK();
        return WCC_OK;
    }
    select_hist_kernel<1><<<grid, SEL_THREADS, 0, st>>>(nrm2, P, k, s.hist, s.state);
    select_hist_kernel<2><<<grid, SEL_THREADS, 0, st>>>(nrm2, P, k, s.hist, s.state);
    select_hist_kernel<3><<<grid, SEL_THREADS, 0, st>>>(nrm2, P, k, s.hist, s.state);
    select_count_kernel<<<grid, SEL_THREADS, 0, st>>>(nrm2, P, s.hist, s.state, s.chunkcnt, tau);
    select_compact_kernel<<<grid, SEL_THREADS, 0, st>>>(nrm2, P, k, s.state, s.chunkcnt, idx, rank, amaxpos, amax_kept);
    g_launches += 4;
    WCC_LAUNCH_CHECK();
    return WCC_OK;
}

}  // namespace wcc
