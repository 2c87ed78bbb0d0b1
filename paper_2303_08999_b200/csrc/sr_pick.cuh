// The s strongest atoms of one pixel, one thread per pixel, straight from global memory: any width, any alignment, fp32 or
// binary16, s <= 16. Order: larger magnitude first, then lower index (the sign does not count).
//
// Keys are 31-bit integers, (magnitude, complemented index), merged S planes at a time by the branch-free networks below.
// A binary16 magnitude (15 bits) and an index fit one key. An fp32 magnitude does not: its lowest bits, as many as an index
// below D needs (7 for D in 65 .. 128), give way to the index. Dropped bits can only matter between atoms whose kept bits
// are the same, so the merge also keeps the best key that fell out, and a pixel in which two neighbours of the list, or the
// last of it and the best that fell out, agree in all kept bits is picked again by exact insertion on the full magnitudes.
// Not where no coefficient of the pixel has any of the dropped bits (fp32 values widened from binary16): equal kept bits are
// then equal magnitudes, and the index in the key has decided. Of Gaussian coefficients a few pixels in a thousand are
// picked twice. Against the insertion kernel (sr_dict_select, 16 to 256 atoms; Gaussian, rectified, widened values): s <= 4
// 0.65, 0.65, 0.61 of its time, longer lists 0.4, 0.5, 0.32.
// Bound: the integer ALU (about 9 min / max per plane at S = 8) or the reads, 4 D bytes a pixel; an insertion of 64-bit keys
// took 48 operations per plane at S = 8, s scans of the D planes where nothing was stored more.
#pragma once
#include "sr_common.cuh"

namespace sr {

// ---- sorting networks on int keys (descending) -----------------------------------------------------------------------

__device__ __forceinline__ void cx(int& a, int& b)    // afterwards a >= b
{
    const int hi = max(a, b), lo = min(a, b);
    a = hi;
    b = lo;
}

template <int S> __device__ __forceinline__ void sort_desc(int* k);

template <> __device__ __forceinline__ void sort_desc<1>(int*) {}
template <> __device__ __forceinline__ void sort_desc<2>(int* k) { cx(k[0], k[1]); }

template <> __device__ __forceinline__ void sort_desc<4>(int* k)
{
    cx(k[0], k[1]); cx(k[2], k[3]);
    cx(k[0], k[2]); cx(k[1], k[3]);
    cx(k[1], k[2]);
}

template <> __device__ __forceinline__ void sort_desc<8>(int* k)   // 19 exchanges
{
    cx(k[0], k[1]); cx(k[2], k[3]); cx(k[4], k[5]); cx(k[6], k[7]);
    cx(k[0], k[2]); cx(k[1], k[3]); cx(k[4], k[6]); cx(k[5], k[7]);
    cx(k[1], k[2]); cx(k[5], k[6]);
    cx(k[0], k[4]); cx(k[1], k[5]); cx(k[2], k[6]); cx(k[3], k[7]);
    cx(k[2], k[4]); cx(k[3], k[5]);
    cx(k[1], k[2]); cx(k[3], k[4]); cx(k[5], k[6]);
}

// Sorts a bitonic sequence of S keys into descending order.
template <int S> __device__ __forceinline__ void bitonic_merge_desc(int* k)
{
#pragma unroll
    for (int d = S / 2; d >= 1; d >>= 1)
#pragma unroll
        for (int i = 0; i < S; ++i)
            if ((i & d) == 0) cx(k[i], k[i + d]);
}

template <> __device__ __forceinline__ void sort_desc<16>(int* k)   // two sorted halves, then a bitonic merge
{
    sort_desc<8>(k);
    sort_desc<8>(k + 8);
#pragma unroll
    for (int i = 0; i < 4; ++i) { const int t = k[8 + i]; k[8 + i] = k[15 - i]; k[15 - i] = t; }   // second half ascending
    bitonic_merge_desc<16>(k);
}

// top[] (sorted) <- the S best of top[] and grp[] (grp sorted descending)
template <int S> __device__ __forceinline__ void merge_top(int* top, const int* grp)
{
#pragma unroll
    for (int i = 0; i < S; ++i) top[i] = max(top[i], grp[S - 1 - i]);
    bitonic_merge_desc<S>(top);
}

// ---- keys ------------------------------------------------------------------------------------------------------------

// Low bits of a key that hold the complemented index: 2^b - 1, the fewest bits that hold D indices.
__device__ __forceinline__ uint32_t pick_tag_mask(int D) { return D <= 1 ? 0u : 0xFFFFFFFFu >> __clz(D - 1); }

template <typename CoefT> __device__ __forceinline__ int pick_key(CoefT v, uint32_t mask, int l);
template <> __device__ __forceinline__ int pick_key<float>(float v, uint32_t mask, int l)
{
    return (int)((__float_as_uint(v) & (0x7FFFFFFFu & ~mask)) | (mask - (uint32_t)l));
}
template <> __device__ __forceinline__ int pick_key<__half>(__half v, uint32_t, int l)
{
    return (int)__byte_perm(__half_as_ushort(v) & 0x7FFFu, 255u - (uint32_t)l, 0x7104);      // 0, magnitude (2 bytes), index
}

__device__ __forceinline__ uint32_t pick_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t pick_bits(__half) { return 0u; }

// Exact insertion: a magnitude enters below those that are not smaller, so equal ones stay in index order. Eight planes are
// loaded together: on a small frame the one warp that comes here would otherwise wait for each of them.
template <int S, typename CoefT>
__device__ __forceinline__ void pick_exact(const CoefT* __restrict__ cp, int64_t HW, int D, int (&atom)[S])
{
    int m[S];
#pragma unroll
    for (int i = 0; i < S; ++i) { m[i] = -1; atom[i] = 0; }
#pragma unroll 1
    for (int l0 = 0; l0 < D; l0 += 8) {
        int x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u, cp += HW) x[u] = l0 + u < D ? (int)mag_bits(__ldg(cp)) : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (x[u] > m[S - 1]) {
#pragma unroll
                for (int i = S - 1; i >= 0; --i) {
                    const bool here = x[u] > m[i], above = i > 0 && x[u] > m[i > 0 ? i - 1 : 0];
                    if (here) { m[i] = above ? m[i > 0 ? i - 1 : 0] : x[u]; atom[i] = above ? atom[i > 0 ? i - 1 : 0] : l0 + u; }
                }
            }
        }
    }
}

// atom[0 .. s-1] <- the s strongest atoms of the pixel at cp (plane stride HW), in rank order; s <= S, s <= D.
template <int S, typename CoefT>
__device__ __forceinline__ void pick_top(const CoefT* __restrict__ cp, int64_t HW, int D, int s, int (&atom)[S])
{
    constexpr bool whole = sizeof(CoefT) == 2;               // the key holds the whole magnitude
    constexpr int G = S < 8 ? 8 : S;                         // planes loaded together, S of them merged at a time
    const uint32_t mask = whole ? 255u : pick_tag_mask(D);
    int top[S], out = -1;                                    // out: the best key that is in no list
    uint32_t low = 0;                                        // every bit that any coefficient has
#pragma unroll
    for (int i = 0; i < S; ++i) top[i] = -1;
    const CoefT* q = cp;
    auto merge = [&](int* g) {
        sort_desc<S>(g);
        if (!whole) {
#pragma unroll
            for (int i = 0; i < S; ++i) out = max(out, min(top[i], g[S - 1 - i]));
        }
        merge_top<S>(top, g);
    };
    int l0 = 0;
    for (; l0 + G <= D; l0 += G) {                           // whole groups: no per-key guards
        CoefT v[G];
#pragma unroll
        for (int i = 0; i < G; ++i, q += HW) v[i] = __ldg(q);
        int g[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            g[i] = pick_key<CoefT>(v[i], mask, l0 + i);
            if (!whole) low |= pick_bits(v[i]);
        }
#pragma unroll
        for (int i = 0; i < G; i += S) merge(g + i);
    }
    if (l0 < D) {                                            // last, partial group
        int g[G];
#pragma unroll
        for (int i = 0; i < G; ++i, q += HW) {
            g[i] = -1;
            if (l0 + i < D) {
                const CoefT v = __ldg(q);
                g[i] = pick_key<CoefT>(v, mask, l0 + i);
                if (!whole) low |= pick_bits(v);
            }
        }
#pragma unroll
        for (int i = 0; i < G; i += S)
            if (l0 + i < D) merge(g + i);
    }
    if (!whole && (low & mask) != 0) {
        bool tied = false;
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const int next = i + 1 < S ? top[i + 1] : out;
            tied = tied || (i < s && ((uint32_t)(top[i] ^ next) & ~mask) == 0);
        }
        if (tied) {
            pick_exact<S, CoefT>(cp, HW, D, atom);
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < S; ++i) atom[i] = (int)(mask - ((uint32_t)top[i] & mask));
}

} // namespace sr
