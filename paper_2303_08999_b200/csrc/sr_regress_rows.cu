// Dense and global-subset regression of binary16 coefficients in rows of any width and alignment:
//   out[c][i] = sum_j (sum_l w_l Phi_l[i] dict_l[j]) B_{i,c}[j]
// The tensor-core layouts copy 16-byte columns of a row and so need widths that are multiples of eight; photographs and
// test images have any width, and consecutive planes of an odd-sized frame even differ in their alignment by half a
// word. This kernel has no roles and no operand in a fixed shared-memory layout: every warp walks rows of 64 pixels on
// its own. A row's pieces of sixteen planes (a K-step) travel through a ring of the warp as the 16-byte chunks that cover
// them; lanes read their words, shift the pixels into place, pair up two planes' values of a pixel, and feed
// mma.sync (m16n8k16) with the coefficients as A (16 pixels x 16 atoms) and the dictionary as B.
//
// Which lane gets which number is chosen for what follows: lane (g, t) (g = lane / 4, t = lane % 4) ends with the filters of
// the eight consecutive pixels 8 g .. 8 g + 7, and of those the taps of patch row t (and its share of the rows beyond
// three; Taps). So it applies them to a window of the up-sampled tile that it reads with 16-byte loads, and four lanes'
// sums make a pixel.
//
// Precision: the dictionary is scaled by a power of two that puts its largest tap near 2^14 and split into three binary16
// numbers (taps down to 2^-15 of the largest enter whole, smaller ones to 2^-39 of it), products are exact, sixteen atoms are
// summed by the tensor core and those sums are added in fp32.
#include <math.h>
#include <type_traits>

#include "sr_regress_rows.cuh"
#include "sr_tile_upsample.cuh"

namespace sr {

namespace {

using namespace tile;

constexpr int kWarps = 4, kNT = 32 * kWarps;
constexpr int TWD = 64;                                  // pixels of a row a warp works on; tile width
constexpr int kRing = 4;                                 // K-steps in a warp's ring
constexpr int kPitch = 36;                               // words of a plane's piece: nine 16-byte chunks
constexpr int kStage = 16 * kPitch;                      // words of a K-step

// Columns of B: lane t's accumulator columns are 2 n + (0, 1) of every n-tile n; column ci of lane t holds this tap.
// K = 3: row t (t < 3). K = 5: row t, then (4, t), then for t = 0 also (4, 4). K = 7: row t, then row t + 4 (t < 3).
template <int K> struct Taps;
template <> struct Taps<3> {
    static constexpr int NT = 2;
    __host__ __device__ static constexpr int of(int t, int ci) { return t < 3 && ci < 3 ? t * 3 + ci : -1; }
};
template <> struct Taps<5> {
    static constexpr int NT = 4;
    __host__ __device__ static constexpr int of(int t, int ci) { return ci < 5 ? t * 5 + ci : (ci == 5 ? 20 + t : (ci == 6 && t == 0 ? 24 : -1)); }
};
template <> struct Taps<7> {
    static constexpr int NT = 7;
    __host__ __device__ static constexpr int of(int t, int ci) { return ci < 7 ? t * 7 + ci : (t < 3 ? (t + 4) * 7 + ci - 7 : -1); }
};

struct RowParams {
    const float* lr;
    const __half* coef;
    const float* dict;
    void* out;
    const uint8_t* idx;   // atom ids of a subset, or nullptr
    const float* gamma;   // its weights, or nullptr
    Geom g;
    int64_t coef_elems;   // elements of the coefficient tensor
    int natoms, ksteps;
    int planes;           // planes per frame in the coefficient tensor
    int gather;           // 1: the subset's planes are planes idx[q] of the full tensor
    int off_b2, off_off, off_u, off_v, off_l, off_ring;   // shared-memory offsets in words
};

__device__ __forceinline__ void cp16(uint32_t dst, uintptr_t src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
// reads `bytes` of the source and zeroes the rest
__device__ __forceinline__ void cp16_part(uint32_t dst, uintptr_t src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma16816_first(float* d, const uint32_t* a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ uint32_t pack_half(__half a, __half b) { return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16); }

// One pixel summed as the other kernels do it: cp its coefficient in plane 0, u the first value of its patch. For pixels whose sum is
// not finite: an infinite coefficient times the parts of a tap, or times the zeros of the columns without one, is not what it
// is times the tap.
template <int K>
__device__ __noinline__ float exact_pixel(const RowParams& p, const int64_t* sOff, const __half* cp, const float* u)
{
    float y = 0.f;
#pragma unroll 1
    for (int j = 0; j < K * K; ++j) {
        float f = 0.f;
#pragma unroll 1
        for (int l = 0; l < p.natoms; ++l) {
            const int a = p.idx ? min((int)__ldg(p.idx + l), p.g.pb.D - 1) : l;
            const float wgt = __half2float(__ldg(cp + sOff[l])) * (p.gamma ? __ldg(p.gamma + l) : 1.f);
            f = fmaf(__ldg(p.dict + (int64_t)a * (K * K) + j), wgt, f);
        }
        y = fmaf(f, u[(j / K) * tile_uw((K - 1) / 2, TWD) + j % K], y);
    }
    return y;
}

// GATHER: the subset's planes are picked one by one out of the full tensor; otherwise a frame's planes follow each other
template <int K, int CTAS, bool GATHER>
__global__ void __launch_bounds__(kNT, CTAS) regress_rows_kernel(const __grid_constant__ RowParams p)
{
    constexpr int kk = K * K, P = (K - 1) / 2, NT = Taps<K>::NT, UW = tile_uw(P, TWD), UW4 = UW / 4;
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ float wpad[kMaxScale][12];
    __shared__ float sMax[kWarps];
    const Geom& g = p.g;
    const Problem& pb = g.pb;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lg = lane >> 2, lt = lane & 3;
    const int C = pb.c, W = pb.W, natoms = p.natoms, ksteps = p.ksteps;
    const int64_t HW = (int64_t)pb.H * W;
    uint4* sB1 = reinterpret_cast<uint4*>(smem);                          // [ksteps][NT][32]: first and second part, two registers each
    uint2* sB2 = reinterpret_cast<uint2*>(smem + p.off_b2);               // [ksteps][NT][32]: third part
    int64_t* sOff = reinterpret_cast<int64_t*>(smem + p.off_off);         // [16 ksteps]: first element of the atom's plane in frame 0
    float* sU = reinterpret_cast<float*>(smem + p.off_u);                 // [C][uh][UW]
    float* sV = reinterpret_cast<float*>(smem + p.off_v);                 // [C][uh][tcols]
    float* sL = reinterpret_cast<float*>(smem + p.off_l);                 // [C * trows][tcols]
    uint32_t* ring = smem + p.off_ring + warp * (kRing * kStage);
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    const int64_t frame_elems = (int64_t)p.planes * HW;
    const uintptr_t begin = reinterpret_cast<uintptr_t>(p.coef), end = reinterpret_cast<uintptr_t>(p.coef + p.coef_elems);

    for (int l = tid; l < 16 * ksteps; l += kNT) {
        const int q = min(l, natoms - 1);
        sOff[l] = (int64_t)(p.gather ? min((int)__ldg(p.idx + q), pb.D - 1) : q) * HW;
    }
    __syncthreads();

    // ---- the warp's copies: its rows are warp, warp + 4, ... of the tiles blockIdx.x, blockIdx.x + gridDim.x, ...; this
    // cursor runs kRing - 1 K-steps ahead of the arithmetic
    int ft = blockIdx.x, fr = warp, fk = 0, ff = 0, fy = 0, fx = 0, frows = 0;
    if (ft < g.num_tiles) decode_tile(g, ft, ff, fy, fx, frows);
    auto settle = [&]() {                                    // to the next row that exists
        while (ft < g.num_tiles && fr >= frows) {
            ft += gridDim.x;
            fr = warp;
            if (ft < g.num_tiles) decode_tile(g, ft, ff, fy, fx, frows);
        }
    };
    settle();
    uint32_t fslot = 0;                                      // byte offset of the slot to fill
    auto fetch = [&]() {
        if (ft < g.num_tiles) {
            const int64_t row = (int64_t)ff * frame_elems + (int64_t)(fy + fr) * W + fx;     // element in plane 0
            // 144 chunks, nine to a plane; a plane's first chunk may begin, its last end, with another row's elements. At
            // the tensor's two ends (its start may lie inside a chunk) only what exists is read.
            const int n = min(16, natoms - 16 * fk);
            const uint32_t dst = ring_s + fslot + 16 * lane;
            if (!GATHER && row >= 8 && row + (int64_t)(natoms - 1) * HW + 72 <= p.coef_elems) {
                const uintptr_t base = reinterpret_cast<uintptr_t>(p.coef + row + (int64_t)(16 * fk) * HW);
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    const int e = lane + 32 * j, q = (e * 57) >> 9, ch = e - 9 * q;          // e / 9, e % 9
                    if (q < n) cp16(dst + 512 * j, ((base + (uintptr_t)(2 * HW) * q) & ~(uintptr_t)15) + 16 * ch);
                }
            } else {
                const uintptr_t base = reinterpret_cast<uintptr_t>(p.coef + row);
                const int64_t* off = sOff + 16 * fk;
                for (int j = 0; j < 5; ++j) {
                    const int e = lane + 32 * j, q = (e * 57) >> 9, ch = e - 9 * q;
                    if (q < n) {
                        const uintptr_t a0 = (base + 2 * off[q]) & ~(uintptr_t)15;
                        const int64_t left = (int64_t)(end - a0) - 16 * ch;
                        const uint32_t bytes = left >= 16 ? 16u : (left > 0 ? (uint32_t)left : 0u);
                        if (a0 + 16 * ch < begin) {          // the one chunk the tensor starts in: element by element
                            for (int u = 0; u < 8; ++u) {
                                const uintptr_t a = a0 + 2 * u;
                                const uint16_t v = a >= begin && a < end ? __ldg(reinterpret_cast<const uint16_t*>(a)) : (uint16_t)0;
                                asm volatile("st.shared.b16 [%0], %1;" ::"r"(dst + 512 * j + 2 * u), "h"(v) : "memory");
                            }
                        } else {
                            cp16_part(dst + 512 * j, a0 + (bytes ? 16 * ch : 0), bytes);
                        }
                    }
                }
            }
            if (++fk == ksteps) {
                fk = 0;
                fr += kWarps;
                settle();
            }
        }
        fslot = fslot + 4 * kStage == 4 * kRing * kStage ? 0 : fslot + 4 * kStage;
        cp_commit();
    };
#pragma unroll
    for (int u = 0; u < kRing - 1; ++u) fetch();

    // ---- set-up: the scaled dictionary in three parts, in the order the lanes want it
    fill_wpad(pb, wpad, tid, kNT);
    for (int i = tid; i < (p.off_ring - p.off_v) / 4; i += kNT) reinterpret_cast<float4*>(sV)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto dict_value = [&](int l, int tap) {
        const int a = p.idx ? min((int)__ldg(p.idx + l), pb.D - 1) : l;
        return __ldg(p.dict + (int64_t)a * kk + tap) * (p.gamma ? __ldg(p.gamma + l) : 1.f);
    };
    float m = 0.f;
#pragma unroll 8
    for (int i = tid; i < natoms * kk; i += kNT) {
        const int l = i / kk;
        m = fmaxf(m, fabsf(dict_value(l, i - l * kk)));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) sMax[warp] = m;
    __syncthreads();
    m = fmaxf(fmaxf(sMax[0], sMax[1]), fmaxf(sMax[2], sMax[3]));
    const int se = m > 0.f ? max(-113, min(126, 14 + 127 - (int)(__float_as_uint(m) >> 23))) : 0;      // (both powers are normal numbers)
    const float scale = __uint_as_float((uint32_t)(127 + se) << 23), unscale = __uint_as_float((uint32_t)(127 - se) << 23);
    for (int i = tid; i < ksteps * NT * 32; i += kNT) {
        const int ln = i & 31, n = (i >> 5) % NT, ks = (i >> 5) / NT;
        const int tap = Taps<K>::of((ln >> 2) >> 1, 2 * n + ((ln >> 2) & 1));        // column ln / 4 of the n-tile
        uint32_t r[3][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            __half part[2][3];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int l = 16 * ks + 2 * (ln & 3) + 8 * h + e;
                float v = tap >= 0 && l < natoms ? dict_value(l, tap) * scale : 0.f;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    part[e][q] = __float2half_rn(v);
                    v -= __half2float(part[e][q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) r[q][h] = pack_half(part[0][q], part[1][q]);
        }
        sB1[i] = make_uint4(r[0][0], r[0][1], r[1][0], r[1][1]);
        sB2[i] = make_uint2(r[2][0], r[2][1]);
    }
    __syncthreads();

    const int tc4 = g.tcols >> 2;
    const int v_lanes = kNT / tc4, v_lane = fast_div(tid, tc4, g.tc4_magic);
    constexpr int kHLanes = kNT / UW4;
    const int h_lane = tid / UW4;
    const bool clamp01 = (pb.flags & SR_CLAMP01) != 0;
    const uint32_t base_mis = (uint32_t)(reinterpret_cast<uintptr_t>(p.coef) >> 1);
    uint32_t slot = 0;                                       // word offset of the slot to read
    LrWindow w;
    {
        decode_tile(g, blockIdx.x, w.f, w.y0, w.x0, w.rows);
        lr_window_of_tile<P, TWD>(g, w);
        prefetch_lr_window_of(g, p.lr, w, sL, tid, kNT);
        cp_commit();
    }
    int since = 0;                                           // K-steps asked for since the LR window was
    for (int tile = blockIdx.x; tile < g.num_tiles; tile += gridDim.x) {
        decode_tile(g, tile, w.f, w.y0, w.x0, w.rows);
        lr_window_of_tile<P, TWD>(g, w);
        // ---- the up-sampled tile
        if (since >= kRing - 1) cp_wait<kRing - 1>();        // the window is older than the ring's copies in flight
        else cp_wait<0>();
        __syncthreads();                                     // it landed for everybody; the previous tile's U is no longer read
        const int uh = w.rows + 2 * P;
        if (v_lane < v_lanes) vertical_pass(g, w, uh, P, sL, sV, (tid - v_lane * tc4) * 4, v_lane, v_lanes);
        __syncthreads();
        since = 0;
        if (tile + (int)gridDim.x < g.num_tiles) {
            LrWindow wn;
            decode_tile(g, tile + gridDim.x, wn.f, wn.y0, wn.x0, wn.rows);
            lr_window_of_tile<P, TWD>(g, wn);
            prefetch_lr_window_of(g, p.lr, wn, sL, tid, kNT);
        }
        cp_commit();
        if (h_lane < kHLanes) horizontal_pass<P, TWD>(g, wpad, w, uh, sV, sU, tid - h_lane * UW4, h_lane, kHLanes);
        __syncthreads();

        for (int r = warp; r < w.rows; r += kWarps) {
            // ---- filters: acc[m-tile i][n-tile][..]; rows lg and lg + 8 of m-tile i are the pixels 8 lg + 2 i, + 1
            const int64_t row = (int64_t)w.f * frame_elems + (int64_t)(w.y0 + r) * W + w.x0;
            const uint32_t row_mis = base_mis + (uint32_t)row;
            // planes eight apart are misaligned alike
            const uint32_t mis2[2] = {(row_mis + (uint32_t)(2 * lt) * (uint32_t)HW) & 7u, (row_mis + (uint32_t)(2 * lt + 1) * (uint32_t)HW) & 7u};
            float acc[4][NT][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[i][n][e] = 0.f;
#pragma unroll 1
            for (int ks = 0; ks < ksteps; ++ks) {
                // the LR window's group, once per tile, sits among the ring's: one more may still travel
                if (since < kRing - 1) cp_wait<kRing - 1>();
                else cp_wait<kRing - 2>();
                __syncwarp();
                uint32_t a[4][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {                // atoms 2 lt, 2 lt + 1 and those eight further on
                    uint32_t v[2][4];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int q = 2 * lt + 8 * h + e;
                        // the piece starts mis halves into its first chunk: two words of that by the address (8-byte loads), a
                        // word and half a word by selects and shifts
                        const uint32_t mis = GATHER ? (row_mis + (uint32_t)sOff[16 * ks + q]) & 7u : mis2[e];
                        const uint32_t* src = ring + slot + q * kPitch + 4 * lg + (mis >> 2) * 2;
                        const uint2 p0 = *reinterpret_cast<const uint2*>(src), p1 = *reinterpret_cast<const uint2*>(src + 2),
                                    p2 = *reinterpret_cast<const uint2*>(src + 4);
                        const bool one = mis & 2u;
                        const uint32_t d0 = one ? p0.y : p0.x, d1 = one ? p1.x : p0.y, d2 = one ? p1.y : p1.x, d3 = one ? p2.x : p1.y, d4 = one ? p2.y : p2.x;
                        const uint32_t sh = (mis & 1u) * 16u;
                        v[e][0] = __funnelshift_r(d0, d1, sh);
                        v[e][1] = __funnelshift_r(d1, d2, sh);
                        v[e][2] = __funnelshift_r(d2, d3, sh);
                        v[e][3] = __funnelshift_r(d3, d4, sh);
                    }
                    if (16 * ks + 16 > natoms) {             // beyond the atoms: what the slot held before
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            if (16 * ks + 2 * lt + 8 * h + e >= natoms) v[e][0] = v[e][1] = v[e][2] = v[e][3] = 0u;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        a[i][2 * h] = __byte_perm(v[0][i], v[1][i], 0x5410);
                        a[i][2 * h + 1] = __byte_perm(v[0][i], v[1][i], 0x7632);
                    }
                }
                __syncwarp();                                // the slot is free
                slot = slot + kStage == kRing * kStage ? 0 : slot + kStage;
                fetch();
                ++since;
                const uint4* b1 = sB1 + (ks * NT) * 32 + lane;
                const uint2* b2 = sB2 + (ks * NT) * 32 + lane;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const uint4 hm = b1[n * 32];
                    const uint2 lo = b2[n * 32];
                    float d[4][4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        mma16816_first(d[i], a[i], lo.x, lo.y);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma16816(d[i], a[i], hm.z, hm.w);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma16816(d[i], a[i], hm.x, hm.y);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[i][n][e] += d[i][e];
                }
            }
            // ---- applied: pixel x = 2 i + h of the lane's eight, column ci = 2 n + j is acc[i][n][2 h + j]
            auto F = [&](int x, int ci) { return acc[x >> 1][ci >> 1][2 * (x & 1) + (ci & 1)]; };
            const int px = w.x0 + 8 * lg + 4 * (lt & 1) + (lt & 2);      // this lane's two pixels in the end
            float finite = 0.f;                              // NaN once a sum is not
#pragma unroll 1
            for (int c = 0; c < C; ++c) {
                const float* u0 = sU + (c * g.uh + r) * UW + 8 * lg;
                float s[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) s[x] = 0.f;
                auto patch_row = [&](const float* src, auto first) {     // K taps from column `first` on, one row of the patch
                    constexpr int C0 = decltype(first)::value, NU = (8 + K - 1 + 3) / 4;
                    float u[4 * NU];
#pragma unroll
                    for (int q = 0; q < NU; ++q) *reinterpret_cast<float4*>(u + 4 * q) = *reinterpret_cast<const float4*>(src + 4 * q);
#pragma unroll
                    for (int b = 0; b < K; ++b)
#pragma unroll
                        for (int x = 0; x < 8; ++x) s[x] = fmaf(F(x, C0 + b), u[x + b], s[x]);
                };
                // (a lane without a tap in a column multiplies some U value by a zero filter)
                patch_row(u0 + min(lt, K - 1) * UW, std::integral_constant<int, 0>{});
                if constexpr (K == 5) {
                    const float* u4 = u0 + 4 * UW;
                    float u[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x) s[x] = fmaf(F(x, 5), u4[lt + x], s[x]);
                    *reinterpret_cast<float4*>(u) = *reinterpret_cast<const float4*>(u4 + 4);
                    *reinterpret_cast<float4*>(u + 4) = *reinterpret_cast<const float4*>(u4 + 8);
#pragma unroll
                    for (int x = 0; x < 8; ++x) s[x] = fmaf(F(x, 6), u[x], s[x]);
                }
                if constexpr (K == 7) patch_row(u0 + min(lt + 4, K - 1) * UW, std::integral_constant<int, 7>{});
                // four lanes hold parts of the same eight pixels: each ends with two whole ones
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float send = (lt & 1) ? s[x] : s[x + 4], keep = (lt & 1) ? s[x + 4] : s[x];
                    s[x] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const float send = (lt & 2) ? s[x] : s[x + 2], keep = (lt & 2) ? s[x + 2] : s[x];
                    s[x] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
                }
                const int64_t o = ((int64_t)w.f * C + c) * HW + (int64_t)(w.y0 + r) * W + px;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    float v = s[x] * unscale;
                    finite = fmaf(v, 0.f, finite);
                    if (clamp01) v = fminf(fmaxf(v, 0.f), 1.f);
                    if (px + x < W) store_out(reinterpret_cast<float*>(p.out), o + x, v, pb.flags);
                }
            }
            if (!(finite == 0.f)) {                          // (here, where the filters' registers are free: called inside the loop, frames of 3 x 3 and
                                                             // 7 x 7 atoms took 8 to 11 % longer; here 0.5 to 3.5 %)
#pragma unroll 1
                for (int j = 0; j < 2 * C; ++j) {
                    const int c = j >> 1, at = px + (j & 1) - w.x0;
                    if (px + (j & 1) >= W) continue;
                    float v = exact_pixel<K>(p, sOff, p.coef + row + at, sU + (c * g.uh + r) * UW + at);
                    if (fabsf(v) * scale < 1e37f) continue;  // a finite one among them: what is stored
                    if (clamp01) v = fminf(fmaxf(v, 0.f), 1.f);
                    store_out(reinterpret_cast<float*>(p.out), ((int64_t)w.f * C + c) * HW + (int64_t)(w.y0 + r) * W + w.x0 + at, v, pb.flags);
                }
            }
        }
    }
    cp_wait<0>();
}

constexpr int kRowsSmemMax = 224 * 1024;
constexpr size_t kSmPool = 228 * 1024;                   // shared memory of an SM
// what a block takes of it: its dynamic part, the kernel's own arrays (400 bytes) and the system's kilobyte, in units of 128
constexpr size_t block_smem(size_t dynamic) { return (dynamic + 400 + 1024 + 127) / 128 * 128; }

// Fills the shared-memory plan for tiles of th rows; returns bytes.
template <int K> size_t plan_rows(RowParams& prm, const Problem& pb, int th)
{
    constexpr int P = (K - 1) / 2, NT = Taps<K>::NT;
    plan_geom(prm.g, pb, th, prm.lr, TWD);
    const Geom& g = prm.g;
    auto up4 = [](int v) { return (v + 3) & ~3; };
    prm.ksteps = (prm.natoms + 15) / 16;
    prm.off_b2 = prm.ksteps * NT * 32 * 4;
    prm.off_off = prm.off_b2 + prm.ksteps * NT * 32 * 2;
    prm.off_u = prm.off_off + 2 * 16 * prm.ksteps;
    prm.off_v = prm.off_u + up4(pb.c * g.uh * tile_uw(P, TWD) + 8);
    prm.off_l = prm.off_v + up4(pb.c * g.uh * g.tcols);
    prm.off_ring = prm.off_l + up4(pb.c * g.trows * g.tcols + 8);
    return (size_t)(prm.off_ring + kWarps * kRing * kStage) * 4;
}

// Blocks per SM the kernel is compiled for.
template <int K> constexpr int blocks_per_sm() { return K == 3 ? 4 : (K == 5 ? 3 : 2); }

// Tile height, geometry and shared memory of a launch; returns bytes (above kRowsSmemMax: the kernel cannot run).
// Rows per warp and tile: three where the taller tile leaves room for all blocks and work for them (213 x 321 x3: 63.2 us
// against 63.8 with two, 71 with one), else two, else one (123 x 129: 15.0 against 19.1).
template <int K> size_t choose_rows(RowParams& prm, const Problem& pb)
{
    constexpr int CTAS = blocks_per_sm<K>();
    for (int rows : {3, 2, 1}) {
        const size_t smem = plan_rows<K>(prm, pb, rows * kWarps);
        if (rows == 1 || (prm.g.num_tiles >= sm_count() * CTAS && (rows == 2 || CTAS * block_smem(smem) <= kSmPool))) return smem;
    }
    return 0;
}

// The kernel's expected time, us. A block works in turns of one tile, x rows per warp in all, 64 columns wide whatever the
// frame's width. Before that the dictionary is laid out, by K-step. A row costs by K-step, by channel, and by channel over the
// scale (the LR image's part of the up-sampled tile), and more of each where other blocks share the SM. Fitted to 2550 of the
// frames that regress_general_us is fitted to (standard deviation 10 to 11 %).
template <int K> struct Cost;
template <> struct Cost<3> { static constexpr float launch = 4.38f, layout = 0.45f, step = 0.35f, step_shared = 0.22f, channel = 0.39f, channel_shared = 0.f, lr = 0.15f, lr_shared = 0.18f; };
template <> struct Cost<5> { static constexpr float launch = 4.65f, layout = 0.88f, step = 1.25f, step_shared = 0.01f, channel = 0.05f, channel_shared = 0.14f, lr = 0.58f, lr_shared = 0.f; };
template <> struct Cost<7> { static constexpr float launch = 4.48f, layout = 2.01f, step = 1.14f, step_shared = 0.f, channel = 0.07f, channel_shared = 0.24f, lr = 0.05f, lr_shared = 0.14f; };

template <int K> float rows_us(int natoms, const Problem& pb)
{
    RowParams prm{};
    prm.natoms = natoms;
    const size_t smem = choose_rows<K>(prm, pb);
    if (smem > (size_t)kRowsSmemMax) return INFINITY;
    const int sms = sm_count(), rows = prm.g.th / kWarps, fit = (int)(kSmPool / block_smem(smem));
    const int blocks = fit < blocks_per_sm<K>() ? fit : blocks_per_sm<K>();
    const int turns = (prm.g.num_tiles + sms * blocks - 1) / (sms * blocks), tiles_per_sm = (prm.g.num_tiles + sms - 1) / sms;
    const float x = (float)(turns * rows), shared = (float)(tiles_per_sm < blocks ? tiles_per_sm : blocks);
    using C = Cost<K>;
    return C::launch + C::layout * prm.ksteps +
           x * (prm.ksteps * (C::step + C::step_shared * shared) + pb.c * (C::channel + C::channel_shared * shared + (C::lr + C::lr_shared * shared) / pb.r));
}

// Infinite where the kernel cannot run or has too few pixels to repay the ring and the dictionary's fragments (rows / thread per
// pixel, us: 9207 px D = 72 k = 3 10.8 / 8.1, k = 5 13.6 / 11.8, D = 128 k = 7 26.5 / 23.8; 21412 px 11.0 / 8.2, 14.0 / 12.0, 27.4 / 24.2).
float estimate(int mode, const Problem& pb)
{
    if ((int64_t)pb.n * pb.H * pb.W < 32768) return INFINITY;
    const int natoms = mode == kModeGlobal ? pb.s : pb.D;
    return pb.k == 3 ? rows_us<3>(natoms, pb) : (pb.k == 5 ? rows_us<5>(natoms, pb) : rows_us<7>(natoms, pb));
}

template <int K, int CTAS, bool GATHER>
cudaError_t launch_g(RowParams& prm, const Problem& pb, cudaStream_t st)
{
    const size_t smem = choose_rows<K>(prm, pb);
    if (smem > (size_t)kRowsSmemMax) return cudaErrorNotSupported;
    auto kern = regress_rows_kernel<K, CTAS, GATHER>;
    static bool configured[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmemMax);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    const int ctas = prm.g.num_tiles < sm_count() * CTAS ? prm.g.num_tiles : sm_count() * CTAS;
    kern<<<ctas, kNT, smem, st>>>(prm);
    count_launches(1);
    return cudaGetLastError();
}

template <int K>
cudaError_t launch_k(RowParams& prm, const Problem& pb, cudaStream_t st)
{
    constexpr int CTAS = blocks_per_sm<K>();
    return prm.gather ? launch_g<K, CTAS, true>(prm, pb, st) : launch_g<K, CTAS, false>(prm, pb, st);
}

} // namespace

bool regress_rows_form(int mode, int coef_dtype, const Problem& pb)
{
    return (mode == kModeDense || mode == kModeGlobal) && coef_dtype == SR_F16 && pb.c <= 4 && !(pb.flags & SR_LUMA_ONLY) &&
           (pb.k == 3 || pb.k == 5 || pb.k == 7);
}

// On the 2550 frames: taken for 1974, 0.73 of the other kernel's time on average; 46 frames lose more than 6 % against that kernel,
// 71 against this one, 46 % at most.
bool regress_rows_pay(int mode, const Problem& pb) { return estimate(mode, pb) < regress_general_us(mode, SR_F16, pb); }

float regress_rows_or_general_us(int mode, const Problem& pb)
{
    const float rows = estimate(mode, pb), general = regress_general_us(mode, SR_F16, pb);
    return rows < general ? rows : general;
}

cudaError_t launch_regress_rows(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma, const float* dict,
                                float* out, const Problem& pb, cudaStream_t st)
{
    RowParams prm{};
    prm.lr = lr; prm.coef = static_cast<const __half*>(coef); prm.dict = dict; prm.out = out;
    if (mode == kModeGlobal) {
        prm.idx = idx; prm.gamma = gamma;
        prm.natoms = pb.s;
        prm.gather = (pb.flags & SR_COEF_COMPACT) ? 0 : 1;
        prm.planes = prm.gather ? pb.D : pb.s;
    } else {
        prm.natoms = prm.planes = pb.D;
    }
    prm.coef_elems = (int64_t)pb.n * prm.planes * pb.H * pb.W;
    switch (pb.k) {
    case 3: return launch_k<3>(prm, pb, st);
    case 5: return launch_k<5>(prm, pb, st);
    case 7: return launch_k<7>(prm, pb, st);
    default: return cudaErrorNotSupported;
    }
}

} // namespace sr
