// Dictionary selection search on the device (Section III-A: Eq. 5-9, Algorithm 1).
//
// The search decides which alpha L of the L atoms a model keeps, and the per-atom re-weights gamma of its coefficient
// layer; its result is what the global-subset mode of sr_dict_regress_selected consumes. Two kernels:
//
//  selection_gram_kernel   Gram statistics over sampled HR pixels (all pixels when no sample list is given): with
//        z_l[i,c] = Phi_l[i] (dict_l . B_{i,c}) the response of atom l alone at pixel i, channel c (Eq. 6 with
//        F_{W,beta} = Phi diag(beta) D), G = Z^T Z, b = Z^T h, hh = h^T h for the target image h. Patches, responses and
//        a register-tiled fp32 rank update, summed in fp64; every CTA leaves its sums in a slot of scratch memory and a
//        second kernel adds the slots in a fixed order (no atomics: results are reproducible).
//  selection_search_kernel   Algorithm 1 on G, b, hh in fp64 by one cluster of thread blocks: LASSO by cyclic coordinate descent
//        (Eq. 7), lambda doubling and bisection to || beta ||_0 ~ alpha_t L, least-squares re-fit of gamma on the
//        support (Eq. 9, Cholesky), gamma folded into G and b, next alpha_t. Every element-wise update and every sum runs
//        in the same order as a sequential program, with separate multiplies and adds (no contraction), so the result
//        does not depend on the parallelisation.
#include <cooperative_groups.h>

#include "sr_common.cuh"
#include "sr_selection.cuh"

namespace sr {

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxSearchL = 128;

// ---- Gram statistics -------------------------------------------------------------------------------------------------
//
// One CTA per SM: a rank group of 192 threads and two producer groups of 160. The producers take the chunks of the CTA
// in turn; a chunk is PX pixels (rows = C PX <= 96 rows of Z, channel-major):
//   1  patches    sPatch[tap][row]: separable up-sampling out of the pixels' LR windows, one thread per patch column
//   2  responses  sZ[row][atom] = Phi * (dict . patch): 8 rows x T atoms per thread, both operands read as float4
// The rank group turns the producers' Z into T x T blocks of the UPPER triangle of Z^T Z, one block per thread, the rows
// dealt over groups of threads. The LR windows of a producer's next chunk travel (cp.async) behind stage 2, its
// coefficients and targets from the end of stage 2 to the next chunk's stage 2: sampled pixels are scattered, every
// coefficient is a 32-byte sector of its own, and that latency has to be covered.
// fp32 only ever sums the terms of 32 pixels, 96 at most: then a thread adds its block to the CTA's fp64 sums, which stay in
// shared memory until the CTA is done.
// Bound: the shared-memory pipe (about 60 % busy) and, beside it, the FMA pipe: a T x T block reads 2 T words for T^2
// multiply-adds, sixteen clocks of either per warp and row at T = 8. 100 000 sampled pixels of a 1080p frame, D = 72,
// k = 5, c = 3: 660 -> 176 us (before: an fp64 read-modify-write of the whole matrix in global memory per 32 pixels, one
// response per thread with scalar loads, sixteen taps per patch element). Also tried: every warp in all three stages, two
// CTAs per SM (304 us); scalar instead of packed multiply-adds with operands loaded a row ahead (226 us); a rank group
// of 256 threads (193 us).
constexpr int kGramRows = 96;          // most rows of Z per chunk, and most terms of an fp32 sum
constexpr int kGramRank = 192;         // threads of the rank group: at least the 136 blocks of 128 atoms
constexpr int kGramProd = 160;         // threads of a producer group
constexpr int kGramThreads = kGramRank + 2 * kGramProd;
constexpr int kGramMaxGroups = 16;
constexpr int kGramSmemMax = 216 * 1024;      // dynamic shared memory of a CTA

struct GramParams {
    const float* lr;
    const void* coef;
    int coef_f16;
    const float* dict;
    const float* target;
    const int64_t* samples;
    int64_t count;            // sampled pixels (or n H W)
    Problem pb;
    double* slots;            // [ctas][Dp * Dp + Dp + 8]
    int Dp;                   // row pitch of a slot's matrix (D rounded up to 16)
    int px, rows;             // pixels and rows per chunk: px a multiple of 4 that divides kGramProd, rows = px * c
    int nb, nblk, groups;     // blocks of T atoms, blocks of the upper triangle, row groups of the rank stage
    int flush_every;          // chunks between two additions to the fp64 sums
    int nw;                   // side of a pixel's LR window
    uint32_t px_magic, nw_magic, nb_magic, r_magic, rows_magic;
    int off_acc, off_set, set_floats;                    // shared-memory offsets in floats: fp64 sums, producer sets
    int off_z, off_h, off_win, off_phi;                  // inside a producer's set (patches first)
};

// floor(x / d) for 0 <= x < 2^29, magic = ceil(2^32 / d)
__device__ __forceinline__ int gram_div(int x, int d, uint32_t magic) { return d == 1 ? x : (int)__umulhi((uint32_t)x, magic); }
__device__ __forceinline__ void gram_cp4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void gram_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void gram_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void gram_bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void gram_bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// named barriers: the rank group, the producers, Z of producer b complete, Z of producer b consumed
enum { kBarRank = 1, kBarProd = 2, kBarFull = 4, kBarEmpty = 6 };

// Column of atom l in a row of Z and in the transposed dictionary: at T = 8 the first and the second four atoms of all
// blocks lie apart, so that neighbouring blocks' 16-byte loads are contiguous (no bank conflicts).
template <int T> __device__ __forceinline__ int gram_col(int l, int nb)
{
    if (T == 4) return l;
    return ((l & 4) ? nb * 4 : 0) + (l >> 3) * 4 + (l & 3);
}

struct __align__(16) GramPixel { int f, pix, Y, X; };                  // f = -1: no pixel

template <int K, int T>
__global__ void __launch_bounds__(kGramThreads, 1) selection_gram_kernel(const __grid_constant__ GramParams p)
{
    constexpr int kk = K * K, P = (K - 1) / 2;
    extern __shared__ __align__(16) float gsm[];
    __shared__ GramPixel sPx[2][2][kGramRows];           // [producer][parity of its chunk count]
    __shared__ __align__(16) int sPar[2][2][kGramRows];  // parity of the pixel's coefficient in plane 0 (which half of a word)
    __shared__ int2 sLo[2][2][kGramRows];                // first LR row / column of its window
    __shared__ float4 sW[kMaxScale];
    __shared__ int sBase[kMaxScale];
    const Problem& pb = p.pb;
    const int C = pb.c, D = pb.D, PX = p.px, rows = p.rows, nb = p.nb, Dz = nb * T, RP = ((rows + 7) & ~7) + 4, r = pb.r, NW = p.nw;
    const int tid = threadIdx.x;
    float* sDict = gsm;                                  // [kk][Dz]
    double* sG = reinterpret_cast<double*>(gsm + p.off_acc);          // [T * T][nblk], then b [Dz], then hh
    double* sB = sG + T * T * p.nblk;
    const int64_t HW = (int64_t)pb.H * pb.W;
    const int hw_odd = (int)(HW & 1);
    const int64_t all_chunks = (p.count + PX - 1) / PX;
    const int chunks = (int)((all_chunks - blockIdx.x + gridDim.x - 1) / gridDim.x);   // of this CTA: blockIdx.x + j gridDim.x

    // ---- set-up
    for (int i = tid; i < T * T * p.nblk + Dz + 1; i += kGramThreads) sG[i] = 0.0;
    for (int i = tid; i < kk * Dz; i += kGramThreads) sDict[i] = 0.f;
    if (tid < kMaxScale) {
        sW[tid] = make_float4(pb.ph.w[tid][0], pb.ph.w[tid][1], pb.ph.w[tid][2], pb.ph.w[tid][3]);
        sBase[tid] = pb.ph.base[tid];
    }
    __syncthreads();
    for (int i = tid; i < D * kk; i += kGramThreads) {
        const int l = i / kk, j = i - l * kk;
        sDict[j * Dz + gram_col<T>(l, nb)] = __ldg(p.dict + i);
    }
    __syncthreads();

    if (tid >= kGramRank) {
        // =================================================================== producers
        const int me = tid >= kGramRank + kGramProd ? 1 : 0, gt = tid - kGramRank - me * kGramProd, warp = gt >> 5, lane = gt & 31;
        float* sPatch = gsm + p.off_set + me * p.set_floats;     // [kk][RP]
        float* sZ = sPatch + p.off_z;                            // [rows][Dz]
        float* sH = sPatch + p.off_h;                            // [2][kGramRows]
        float* sWin = sPatch + p.off_win;                        // [rows][NW * NW]
        uint32_t* sPhi = reinterpret_cast<uint32_t*>(sPatch + p.off_phi);   // phi_at(l, px): the 4-byte word that holds the coefficient
        const int nw2 = NW * NW;
        const uintptr_t coef_base = reinterpret_cast<uintptr_t>(p.coef);
        const uintptr_t coef_end = coef_base + (uintptr_t)((int64_t)pb.n * D * HW) * (p.coef_f16 ? 2 : 4);
        // [D][PX] with four words more after every eighth atom: the eight atoms apart that stage 2's lanes ask for at once
        // start in different 16-byte bank groups
        auto phi_at = [&](int l, int px) { return sPhi + l * PX + ((l >> 3) << 2) + px; };
        auto first_tap = [&](int Zc, int& phase) {               // first LR tap of the (clamped) HR coordinate Zc, and its phase
            const int q = gram_div(Zc, r, p.r_magic);
            phase = Zc - q * r;
            return q + sBase[phase];
        };
        auto load_pixels = [&](int j, int buf) {                 // pixels of this CTA's chunk j
            if (gt >= PX) return;
            const int64_t si = ((int64_t)blockIdx.x + (int64_t)j * gridDim.x) * PX + gt;
            int64_t flat = -1;
            if (j < chunks && si < p.count) flat = p.samples ? __ldg(p.samples + si) : si;
            GramPixel g;
            g.f = -1; g.pix = 0;
            if (flat >= 0 && flat < (int64_t)pb.n * HW) {
                g.f = (int)(flat / HW);
                g.pix = (int)(flat - (int64_t)g.f * HW);
            }
            g.Y = g.pix / pb.W;
            g.X = g.pix - g.Y * pb.W;
            int ph;
            sPx[me][buf][gt] = g;
            sPar[me][buf][gt] = ((int)(coef_base >> 1) + (g.f & D & hw_odd) + g.pix) & 1;
            sLo[me][buf][gt] = make_int2(first_tap(clampi(g.Y - P, 0, pb.H - 1), ph), first_tap(clampi(g.X - P, 0, pb.W - 1), ph));
        };
        auto fetch_windows = [&](int buf) {                      // a warp takes the windows of a pixel in all channels
            const int hw = pb.h * pb.w;
            for (int e = lane; e < nw2; e += 32) {
                const int j = gram_div(e, NW, p.nw_magic), i = e - j * NW;
                for (int px = warp; px < PX; px += kGramProd / 32) {
                    const int f = sPx[me][buf][px].f;
                    const int2 lo = sLo[me][buf][px];
                    float* dst = sWin + px * nw2 + e;
                    const float* src = p.lr + (int64_t)(f * C) * hw + clampi(lo.x + j, 0, pb.h - 1) * pb.w + clampi(lo.y + i, 0, pb.w - 1);
                    if (f >= 0) {
                        for (int c = 0; c < C; ++c) gram_cp4(dst + c * PX * nw2, src + (int64_t)c * hw);
                    } else {
                        for (int c = 0; c < C; ++c) dst[c * PX * nw2] = 0.f;
                    }
                }
            }
            gram_commit();
        };
        auto fetch_coefficients = [&](int buf) {                 // and the targets, into half `buf` of sH; a thread keeps its pixel
            const int l0 = gram_div(gt, PX, p.px_magic), px = gt - l0 * PX, dl = gram_div(kGramProd, PX, p.px_magic);
            const GramPixel g = sPx[me][buf][px];
            if (g.f >= 0) {
                const int64_t elem = ((int64_t)g.f * D + l0) * HW + g.pix;
                if (p.coef_f16) {
                    uintptr_t a = coef_base + (uintptr_t)elem * 2;
#pragma unroll 4
                    for (int l = l0; l < D; l += dl, a += (uintptr_t)(2 * HW) * dl) {
                        const uintptr_t word = a & ~(uintptr_t)3;
                        if (word >= coef_base && word + 4 <= coef_end) {
                            gram_cp4(phi_at(l, px), reinterpret_cast<const void*>(word));
                        } else {                                 // the first or last element, where the word reaches outside the tensor
                            const uint32_t v = __ldg(reinterpret_cast<const unsigned short*>(a));
                            *phi_at(l, px) = v << (8 * (int)(a & 2));
                        }
                    }
                } else {
                    const float* a = reinterpret_cast<const float*>(p.coef) + elem;
#pragma unroll 4
                    for (int l = l0; l < D; l += dl, a += HW * dl) gram_cp4(phi_at(l, px), a);
                }
                for (int c = l0; c < C; c += dl) gram_cp4(sH + buf * kGramRows + c * PX + px, p.target + ((int64_t)g.f * C + c) * HW + g.pix);
            } else {
                for (int l = l0; l < D; l += dl) *phi_at(l, px) = 0u;
                for (int c = l0; c < C; c += dl) sH[buf * kGramRows + c * PX + px] = 0.f;
            }
            gram_commit();
        };

        int buf = 0;
        load_pixels(me, 0);
        gram_bar_sync(kBarProd + me, kGramProd);
        fetch_windows(0);
        fetch_coefficients(0);
        load_pixels(me + 2, 1);
        for (int j = me; j < chunks; j += 2, buf ^= 1) {
            gram_wait<1>();
            gram_bar_sync(kBarProd + me, kGramProd);             // windows landed; the next chunk's pixels are known
            // ---- stage 1: thread = one column of one row's patch; four horizontally filtered window rows slide down
            for (int e = gt; e < rows * K; e += kGramProd) {
                const int b = gram_div(e, rows, p.rows_magic), row = e - b * rows;
                const int c = gram_div(row, PX, p.px_magic), px = row - c * PX;
                const GramPixel g = sPx[me][buf][px];
                const int2 lo = sLo[me][buf][px];
                int phx;
                const int xo = first_tap(clampi(g.X + b - P, 0, pb.W - 1), phx) - lo.y;
                const float4 wx = sW[phx];
                const float* win = sWin + row * nw2 + xo;
                auto hor = [&](int i) {
                    const float* s = win + i * NW;
                    return fmaf(wx.w, s[3], fmaf(wx.z, s[2], fmaf(wx.y, s[1], wx.x * s[0])));
                };
                float t0 = hor(0), t1 = hor(1), t2 = hor(2), t3 = hor(3);
                int cur = 0;
#pragma unroll
                for (int a = 0; a < K; ++a) {
                    int phy;
                    const int yo = first_tap(clampi(g.Y + a - P, 0, pb.H - 1), phy) - lo.x;
                    if (yo > cur) {                              // by one: consecutive HR rows
                        cur = yo;
                        t0 = t1; t1 = t2; t2 = t3;
                        t3 = hor(cur + 3);
                    }
                    const float4 wy = sW[phy];
                    sPatch[(a * K + b) * RP + row] = fmaf(wy.w, t3, fmaf(wy.z, t2, fmaf(wy.y, t1, wy.x * t0)));
                }
            }
            gram_wait<0>();
            gram_bar_sync(kBarProd + me, kGramProd);             // patches complete, coefficients landed, windows consumed
            fetch_windows(buf ^ 1);
            if (j >= 2) gram_bar_sync(kBarEmpty + me, kGramRank + kGramProd);   // the rank group is done with this producer's last Z
            // ---- stage 2: 8 rows x T atoms
            for (int e = gt; e < ((rows + 7) >> 3) * nb; e += kGramProd) {
                const int rg = gram_div(e, nb, p.nb_magic), t = e - rg * nb;
                float2 z[8][T / 2];
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int q = 0; q < T / 2; ++q) z[i][q] = make_float2(0.f, 0.f);
                const float* pp = sPatch + rg * 8;
                const float* dp = sDict + t * 4;
#pragma unroll 5
                for (int i = 0; i < kk; ++i) {
                    float pv[8];
                    *reinterpret_cast<float4*>(pv) = *reinterpret_cast<const float4*>(pp + i * RP);
                    *reinterpret_cast<float4*>(pv + 4) = *reinterpret_cast<const float4*>(pp + i * RP + 4);
                    float2 dv[T / 2];
                    *reinterpret_cast<float4*>(dv) = *reinterpret_cast<const float4*>(dp + i * Dz);
                    if (T == 8) *reinterpret_cast<float4*>(dv + T / 2 - 2) = *reinterpret_cast<const float4*>(dp + i * Dz + nb * 4);
#pragma unroll
                    for (int u = 0; u < 8; ++u)
#pragma unroll
                        for (int q = 0; q < T / 2; ++q) z[u][q] = __ffma2_rn(make_float2(pv[u], pv[u]), dv[q], z[u][q]);
                }
#pragma unroll
                for (int half = 0; half < 2; ++half) {           // four rows of one channel each
                    const int row0 = rg * 8 + 4 * half;
                    if (row0 < rows) {
                        const int px0 = row0 - gram_div(row0, PX, p.px_magic) * PX;
                        const int4 par = *reinterpret_cast<const int4*>(&sPar[me][buf][px0]);
#pragma unroll
                        for (int q = 0; q < T / 4; ++q) {        // atoms 4 q .. 4 q + 3 of the block
                            float o[4][4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int l = t * T + 4 * q + u;
                                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                                if (l < D) w = *reinterpret_cast<const uint4*>(phi_at(l, px0));
                                float f0, f1, f2, f3;
                                if (p.coef_f16) {
                                    const int odd = l & hw_odd;
                                    f0 = __half2float(__ushort_as_half((unsigned short)(w.x >> (16 * (par.x ^ odd)))));
                                    f1 = __half2float(__ushort_as_half((unsigned short)(w.y >> (16 * (par.y ^ odd)))));
                                    f2 = __half2float(__ushort_as_half((unsigned short)(w.z >> (16 * (par.z ^ odd)))));
                                    f3 = __half2float(__ushort_as_half((unsigned short)(w.w >> (16 * (par.w ^ odd)))));
                                } else {
                                    f0 = __uint_as_float(w.x); f1 = __uint_as_float(w.y); f2 = __uint_as_float(w.z); f3 = __uint_as_float(w.w);
                                }
                                o[0][u] = f0 * ((u & 1) ? z[4 * half + 0][2 * q + u / 2].y : z[4 * half + 0][2 * q + u / 2].x);
                                o[1][u] = f1 * ((u & 1) ? z[4 * half + 1][2 * q + u / 2].y : z[4 * half + 1][2 * q + u / 2].x);
                                o[2][u] = f2 * ((u & 1) ? z[4 * half + 2][2 * q + u / 2].y : z[4 * half + 2][2 * q + u / 2].x);
                                o[3][u] = f3 * ((u & 1) ? z[4 * half + 3][2 * q + u / 2].y : z[4 * half + 3][2 * q + u / 2].x);
                            }
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                *reinterpret_cast<float4*>(sZ + (row0 + i) * Dz + q * nb * 4 + t * 4) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
                        }
                    }
                }
            }
            __threadfence_block();                               // (bar.arrive orders nothing by itself for the reader's loads)
            gram_bar_arrive(kBarFull + me, kGramRank + kGramProd);      // Z (and the targets) of this chunk are complete
            gram_bar_sync(kBarProd + me, kGramProd);             // coefficients consumed
            fetch_coefficients(buf ^ 1);
            load_pixels(j + 4, buf);                             // this chunk's pixels are no longer needed
        }
        gram_wait<0>();
    } else {
        // =================================================================== rank update
        const int grp = tid / p.nblk, blk = tid - grp * p.nblk;
        const bool has_block = grp < p.groups;
        int ti = 0, tj = blk;
        while (tj >= nb - ti) { tj -= nb - ti; ++ti; }
        tj += ti;
        float2 acc[T][T / 2];
        float bacc[T], hacc = 0.f;
#pragma unroll
        for (int a = 0; a < T; ++a) {
            bacc[a] = 0.f;
#pragma unroll
            for (int b = 0; b < T / 2; ++b) acc[a][b] = make_float2(0.f, 0.f);
        }
        int since_flush = 0;
        for (int j = 0; j < chunks; ++j) {
            const int b2 = j & 1;
            const float* sZ = gsm + p.off_set + b2 * p.set_floats + p.off_z;
            const float* h = gsm + p.off_set + b2 * p.set_floats + p.off_h + ((j >> 1) & 1) * kGramRows;
            gram_bar_sync(kBarFull + b2, kGramRank + kGramProd);
            if (has_block) {
#pragma unroll 2
                for (int row = grp; row < rows; row += p.groups) {
                    const float* zr = sZ + row * Dz;
                    float za[T];
                    float2 zb[T / 2];
                    *reinterpret_cast<float4*>(za) = *reinterpret_cast<const float4*>(zr + ti * 4);
                    *reinterpret_cast<float4*>(zb) = *reinterpret_cast<const float4*>(zr + tj * 4);
                    if (T == 8) {
                        *reinterpret_cast<float4*>(za + T - 4) = *reinterpret_cast<const float4*>(zr + nb * 4 + ti * 4);
                        *reinterpret_cast<float4*>(zb + T / 2 - 2) = *reinterpret_cast<const float4*>(zr + nb * 4 + tj * 4);
                    }
#pragma unroll
                    for (int a = 0; a < T; ++a)
#pragma unroll
                        for (int b = 0; b < T / 2; ++b) acc[a][b] = __ffma2_rn(make_float2(za[a], za[a]), zb[b], acc[a][b]);
                    if (ti == tj) {
                        const float hv = h[row];
#pragma unroll
                        for (int a = 0; a < T; ++a) bacc[a] = fmaf(za[a], hv, bacc[a]);
                        hacc = fmaf(hv, hv, hacc);
                    }
                }
            }
            if (j + 2 < chunks) gram_bar_arrive(kBarEmpty + b2, kGramRank + kGramProd);
            if (++since_flush >= p.flush_every || j + 1 == chunks) {
                since_flush = 0;
                // fp32 blocks into the fp64 sums. The groups hold partial sums of the same blocks: in step q group g adds
                // row (g + q) mod m of its block, so that all groups work at once, never on the same row, and every
                // sum is formed in a fixed order.
                const int m = max(p.groups, T);
                int want = grp;
                for (int q = 0; q < m; ++q) {
                    if (has_block) {
#pragma unroll
                        for (int a = 0; a < T; ++a) {
                            if (a == want) {
                                double v[T];
#pragma unroll
                                for (int b = 0; b < T; ++b) v[b] = sG[(a * T + b) * p.nblk + blk];
#pragma unroll
                                for (int b = 0; b < T / 2; ++b) {
                                    v[2 * b] += (double)acc[a][b].x;
                                    v[2 * b + 1] += (double)acc[a][b].y;
                                    acc[a][b] = make_float2(0.f, 0.f);
                                }
#pragma unroll
                                for (int b = 0; b < T; ++b) sG[(a * T + b) * p.nblk + blk] = v[b];
                                if (ti == tj) {
                                    sB[ti * T + a] += (double)bacc[a];
                                    bacc[a] = 0.f;
                                    if (ti == 0 && a == 0) { sB[Dz] += (double)hacc; hacc = 0.f; }
                                }
                            }
                        }
                    }
                    if (++want == m) want = 0;
                    gram_bar_sync(kBarRank, kGramRank);
                }
            }
        }
        // ---- the CTA's slot: the upper triangle (block rows ti <= tj, whole blocks on the diagonal), b, hh
        double* slot = p.slots + (int64_t)blockIdx.x * (p.Dp * p.Dp + p.Dp + 8);
        if (grp == 0) {
#pragma unroll
            for (int a = 0; a < T; ++a)
#pragma unroll
                for (int b = 0; b < T; ++b) slot[(ti * T + a) * p.Dp + tj * T + b] = sG[(a * T + b) * p.nblk + blk];
        }
        for (int i = tid; i < D; i += kGramRank) slot[p.Dp * p.Dp + i] = sB[i];
        if (tid == 0) slot[p.Dp * p.Dp + p.Dp] = sB[Dz];
    }
}

// Adds the slots in a fixed order: 32 elements per block, eight threads per element take every eighth slot, their sums
// are added one after the other.
constexpr int kReduceLanes = 8;
__global__ void __launch_bounds__(32 * kReduceLanes) selection_gram_reduce_kernel(const double* slots, int nslots, int Dp, int D, double* G, double* b, double* hh)
{
    __shared__ double part[kReduceLanes][32];
    const int slot_doubles = Dp * Dp + Dp + 8;
    const int total = D * D + D + 1;
    const int i = blockIdx.x * 32 + threadIdx.x;
    int src = -1;
    if (i < D * D) {
        const int row = i / D, col = i - row * D;
        src = min(row, col) * Dp + max(row, col);         // only the upper triangle is in the slots
    } else if (i < D * D + D) {
        src = Dp * Dp + (i - D * D);
    } else if (i < total) {
        src = Dp * Dp + Dp;
    }
    double v = 0.0;
    if (src >= 0) {
#pragma unroll 8
        for (int s = threadIdx.y; s < nslots; s += kReduceLanes) v += slots[(int64_t)s * slot_doubles + src];
    }
    part[threadIdx.y][threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.y == 0 && src >= 0) {
        for (int q = 1; q < kReduceLanes; ++q) v += part[q][threadIdx.x];
        if (i < D * D) G[i] = v;
        else if (i < D * D + D) b[i - D * D] = v;
        else *hh = v;
    }
}

template <int K, int T>
cudaError_t launch_gram_kt(const GramParams& p, int ctas, size_t smem, cudaStream_t st)
{
    auto kern = selection_gram_kernel<K, T>;
    static bool configured[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramSmemMax);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    kern<<<ctas, kGramThreads, smem, st>>>(p);
    count_launches(1);
    return cudaGetLastError();
}

template <int K>
cudaError_t launch_gram_k(const GramParams& p, int T, int ctas, size_t smem, cudaStream_t st)
{
    return T == 4 ? launch_gram_kt<K, 4>(p, ctas, smem, st) : launch_gram_kt<K, 8>(p, ctas, smem, st);
}

// ---- Algorithm 1 in one cluster of thread blocks ------------------------------------------------------------------------
//
// The sweeps of coordinate descent are one serial chain in fp64: coordinate l's step needs the residual that coordinate
// l - 1's step left. One warp walks it; four warps share what is parallel (residuals, factorisation, re-scaling).
// The active atoms are kept compacted (index 0 .. na - 1, order of the atoms), so no step ever looks at a dropped one.
//
// What bounds a sweep is the latency of that chain, so everything else is kept off it. Lane m holds the residuals of
// coordinates m, m + 32, ...; all lanes make every step redundantly. The residual a step needs reaches them by a shuffle that
// leaves two steps earlier, and gets the last step's change in every lane: no shuffle and no load stands between two
// steps. A step is then six dependent fp64 operations: two additions to the thresholded numerator, one
// multiply-add for the quotient, one addition for the step, a product and a sum to the next residual. Every rounding is that
// of the sequential program, so the results are the same bits.
//
// The bisection's solves all start from the same coefficients until one of them is kept. So each round solves the whole
// tree of the next five mid points, one per warp of a cluster of eight blocks (a warp per scheduler: nobody slows the
// chains down), and then walks it as the sequential program would. The blocks run everything else alike. Where the context has no
// room for a cluster of eight, fewer blocks walk shallower trees: the same solves one round later, the same bits.
// 72 atoms down to 8 in four steps (about 90 solves, 90 000 steps, 33 000 of them in bisections): 8.7 -> 6.0 ms against one block
// with eleven operations to a step, a bisection's solves one after the other (46 ms with one warp that divided inside the chain).
// A round lasts as long as its slowest solve, which costs what a walk that ends early saves: 187 searches of 16 to 128 atoms, eps from
// 0 to 2 / L, took 0.84 of that block's time on average, none longer (0.95 to 0.97 with 128 atoms and eps = 2 / L).
// Left are some 165 clocks a step: about 60 instructions of one warp, fp64 at two clocks each, around a chain of 75.
constexpr int kSearchThreads = 128;
constexpr int kSearchWarps = kSearchThreads / 32;
constexpr int kSearchCtas = 8;                     // blocks of the cluster, at most: 31 of the 32 warps have a node of five levels
constexpr int kCdBlock = 8;

struct SearchParams {
    const double* G;
    const double* b;
    const double* hh;
    int L;
    double nrows, alpha, dalpha, eps, lambda0, tol;
    int max_sweeps, max_bisect, max_steps;
    uint8_t* idx_out;
    float* gamma_out;
    int* count_out;
    double* trace;
    int* steps_out;
};

struct SearchState {
    double* G;            // [L8][Lp], active atoms only; rows and columns na .. na8 - 1 are zero
    double* A;            // packed lower triangle
    double *b, *beta, *r, *best, *gtot, *tmp, *prod;
    double *diag, *rcp, *rcl, *frz;  // G[l][l], 1 / G[l][l] rounded and what the rounding left of it, and 0 or (atoms whose G[l][l] is not
                                     // positive: never moved) infinity
    double* sub;          // G[l + 1][l]; of the last coordinate G[0][na8 - 1]
    double* solve;        // [warps][2][L8]: a warp's coefficients, old and new ones of a sweep
    int *S, *orig;        // support; compact index -> atom
    int L8, Lp, na, na8, tid, lane;
    double nrows;
    bool safe;            // every positive G[l][l] lies in [2^-300, 2^300]
    bool frozen;          // some G[l][l] is not positive
};

__host__ __device__ constexpr int search_l8(int L) { return (L + kCdBlock - 1) / kCdBlock * kCdBlock; }

__device__ int count_nonzero(const SearchState& s, const double* beta)   // every warp counts for itself
{
    int n = 0;
    for (int l = s.lane; l < s.na; l += 32) n += beta[l] != 0.0 ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    return n;
}

// Diagonal, reciprocals and padding of the compacted matrix and vectors. Ends in a barrier.
__device__ void prepare_active(SearchState& s)
{
    s.na8 = search_l8(s.na);
    int bad = 0, dead = 0;
    for (int l = s.tid; l < s.L8; l += kSearchThreads) {
        const double g = l < s.na ? s.G[l * s.Lp + l] : 0.0;
        const bool live = g > 0.0;
        const double y = live ? __drcp_rn(g) : 0.0;
        s.diag[l] = g;
        s.rcp[l] = y;
        s.rcl[l] = live ? __dmul_rn(__fma_rn(-g, y, 1.0), y) : 0.0;
        s.frz[l] = live ? 0.0 : __longlong_as_double(0x7FF0000000000000ll);
        if (live && !(g >= 0x1p-300 && g <= 0x1p300)) bad = 1;
        if (l < s.na && !live) dead = 1;
        if (l >= s.na) s.beta[l] = s.best[l] = s.r[l] = 0.0;
        for (int m = l < s.na ? s.na : 0; m < s.na8; ++m) s.G[l * s.Lp + m] = 0.0;
    }
    s.safe = !__syncthreads_or(bad);
    s.frozen = __syncthreads_or(dead);
    for (int l = s.tid; l < s.na8; l += kSearchThreads) s.sub[l] = s.G[(l + 1 < s.na8 ? l + 1 : 0) * s.Lp + l];
    __syncthreads();
}

// The plain form: one warp, sweeps over the active atoms until no coefficient moves by more than tol, quotients by division.
// beta in place; rr: residuals of the coordinates lane, lane + 32, ... Returns the sweeps made; *settled says whether the last one
// moved nothing.
__device__ __noinline__ int cd_sweeps_plain(const SearchState& s, double thr, double (&rr)[4], double* beta, double tol, int max_sweeps, bool* settled)
{
    const int Lp = s.Lp;
    const double* row[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) row[k] = s.G + min(s.lane + 32 * k, s.L8 - 1) * Lp;
    int sweep = 0;
    *settled = false;
    while (sweep < max_sweeps && !*settled) {
        double moved = 0.0;
#pragma unroll 1
        for (int l = 0; l < s.na; ++l) {
            double rk = rr[0];
#pragma unroll
            for (int k = 1; k < 4; ++k) rk = l >= 32 * k ? rr[k] : rk;
            const double g = s.diag[l], be = beta[l], fz = s.frz[l];
            const double rho = __dadd_rn(__shfl_sync(0xffffffffu, rk, l & 31), __dmul_rn(g, be));
            const double nb = fabs(rho) > __dadd_rn(thr, fz) ? __ddiv_rn(__dadd_rn(rho, -copysign(thr, rho)), g) : (fz > 0.0 ? be : 0.0);
            const double d = __dadd_rn(nb, -be);
#pragma unroll
            for (int k = 0; k < 4; ++k) rr[k] = __dadd_rn(rr[k], -__dmul_rn(d, row[k][l]));
            moved = fmax(moved, fabs(d));
            __syncwarp();
            if (s.lane == 0) beta[l] = nb;
            __syncwarp();
        }
        ++sweep;
        *settled = moved <= tol;
    }
    return sweep;
}

__device__ __forceinline__ double with_sign_of(double magnitude, double x)   // magnitude >= 0
{
    return __hiloint2double((__double2hiint(x) & 0x80000000) | __double2hiint(magnitude), __double2loint(magnitude));
}

// One warp; coefficients in buf[0 .. L8), scratch behind them; residuals from s.r. Returns where the coefficients ended up.
//
// The quotient num / g, rounded to nearest, is made as q = num y + t with y the rounded reciprocal and t = num (1/g - y), which is known
// no later than num (from the two terms of num: they cancel where the residual barely exceeds the threshold, and t keeps their rounding).
// That is the rounded quotient but where the quotient lies within about 2^-52 max(1, thr / |num|) units in the last place of the
// middle of two numbers. So every q is checked, off the chain: with the remainder of q, q + remainder y rounds to the
// rounded quotient if q is one of the quotient's two neighbours (Markstein, IBM J. Res. Dev. 34 (1990)), and it differs from q if q
// is further off (or if anything over- or underflowed). A sweep with a q that fails is made again in the plain form, from the
// coefficients and residuals it started with.
template <int NK, bool FROZEN>
__device__ __noinline__ double* cd_sweeps(const SearchState& s, double thr, double* buf, double tol, int max_sweeps)
{
    const int na8 = s.na8;
    double rr[NK];
    const double* row[NK];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int m = s.lane + 32 * k;
        rr[k] = m < na8 ? s.r[m] : 0.0;
        row[k] = s.G + min(m, s.L8 - 1) * s.Lp;
    }
    double *cur = buf, *nxt = buf + s.L8;
    // residuals of this step's coordinate and, without the last step, the next one's
    double r0 = s.r[0], r1 = s.r[1];
#pragma unroll 1
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        double was[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) was[k] = rr[k];
        bool moved = false, bad = false;
#pragma unroll 1
        for (int l0 = 0; l0 < na8; l0 += kCdBlock) {
            auto load = [](double (&to)[kCdBlock], const double* from) {
#pragma unroll
                for (int i = 0; i < kCdBlock; i += 2) {
                    const double2 v = *reinterpret_cast<const double2*>(from + i);
                    to[i] = v.x;
                    to[i + 1] = v.y;
                }
            };
            double g[kCdBlock], y[kCdBlock], yl[kCdBlock], be[kCdBlock], sub[kCdBlock], nb[kCdBlock];
            load(g, s.diag + l0);
            load(be, cur + l0);
            load(y, s.rcp + l0);
            load(yl, s.rcl + l0);
            load(sub, s.sub + l0);
            const int next = l0 + kCdBlock < na8 ? l0 + kCdBlock : 0;
#pragma unroll
            for (int i = 0; i < kCdBlock; ++i) {
                const double rho = __dadd_rn(r0, __dmul_rn(g[i], be[i]));
                const double num = __dadd_rn(rho, -with_sign_of(thr, rho));
                const double tl = __dmul_rn(thr, yl[i]);
                const double t = __fma_rn(rho, yl[i], __hiloint2double((__double2hiint(rho) & 0x80000000) ^ 0x80000000 ^ __double2hiint(tl), __double2loint(tl)));
                const double q = __fma_rn(num, y[i], t);
                bool in = fabs(rho) > thr;
                double out = 0.0;
                if (FROZEN) {
                    const bool held = s.frz[l0 + i] > 0.0;
                    in = in & !held;
                    out = held ? be[i] : 0.0;
                }
                const double d = in ? __dadd_rn(q, -be[i]) : __dadd_rn(out, -be[i]);
                r0 = __dadd_rn(r1, -__dmul_rn(d, sub[i]));
                nb[i] = in ? q : out;
                const double again = __fma_rn(__fma_rn(-g[i], q, num), y[i], q);
                bad = bad | (in & !(again == q));
                moved = moved | (fabs(d) > tol);
#pragma unroll
                for (int k = 0; k < NK; ++k) rr[k] = __dadd_rn(rr[k], -__dmul_rn(d, row[k][l0 + i]));
                const int after = i + 2 < kCdBlock ? l0 + i + 2 : next + i + 2 - kCdBlock;
                double v = rr[0];
#pragma unroll
                for (int k = 1; k < NK; ++k) v = after >= 32 * k ? rr[k] : v;
                r1 = __shfl_sync(0xffffffffu, v, after & 31);
            }
            if (s.lane == 0) {
#pragma unroll
                for (int i = 0; i < kCdBlock; i += 2) *reinterpret_cast<double2*>(nxt + l0 + i) = make_double2(nb[i], nb[i + 1]);
            }
        }
        __syncwarp();
        if (bad) {                                           // the same in every lane
            double again[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 0; k < NK; ++k) again[k] = was[k];
            for (int l = s.lane; l < na8; l += 32) nxt[l] = cur[l];
            __syncwarp();
            bool settled;
            cd_sweeps_plain(s, thr, again, nxt, tol, 1, &settled);
#pragma unroll
            for (int k = 0; k < NK; ++k) rr[k] = again[k];
            r0 = __shfl_sync(0xffffffffu, rr[0], 0);
            r1 = __shfl_sync(0xffffffffu, rr[0], 1);
            moved = !settled;
        }
        double* swap = cur; cur = nxt; nxt = swap;
        if (!moved && tol == tol) break;
    }
    return cur;
}

// s.r = b - G beta; all threads, ends in a barrier.
__device__ void residuals(const SearchState& s, const double* beta)
{
    for (int l = s.tid; l < s.na; l += kSearchThreads) {
        double acc = 0.0;
#pragma unroll 8
        for (int m = 0; m < s.na; ++m) acc = __dadd_rn(acc, __dmul_rn(s.G[l * s.Lp + m], beta[m]));
        s.r[l] = __dadd_rn(s.b[l], -acc);
    }
    __syncthreads();
}

// Eq. 7 by cyclic coordinate descent from `start`, whose residuals are in s.r, by one warp in its own buffers. Same operation
// order as a sequential loop over the atoms. Returns the coefficients.
__device__ double* lasso_cd(const SearchState& s, double lambda, const double* start, double tol, int max_sweeps)
{
    double* buf = s.solve + (s.tid >> 5) * 2 * s.L8;
    for (int l = s.lane; l < s.na8; l += 32) { buf[l] = start[l]; buf[s.L8 + l] = 0.0; }
    __syncwarp();
    const double thr = __dmul_rn(__dmul_rn(0.5, lambda), s.nrows);
    if (s.safe && thr >= 0x1p-300 && thr <= 0x1p300) {
        if (s.frozen) return cd_sweeps<4, true>(s, thr, buf, tol, max_sweeps);
        if (s.na8 <= 32) return cd_sweeps<1, false>(s, thr, buf, tol, max_sweeps);
        if (s.na8 <= 64) return cd_sweeps<2, false>(s, thr, buf, tol, max_sweeps);
        if (s.na8 <= 96) return cd_sweeps<3, false>(s, thr, buf, tol, max_sweeps);
        return cd_sweeps<4, false>(s, thr, buf, tol, max_sweeps);
    }
    double rr[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) rr[k] = s.lane + 32 * k < s.na ? s.r[s.lane + 32 * k] : 0.0;
    bool settled;
    cd_sweeps_plain(s, thr, rr, buf, tol, max_sweeps, &settled);
    return buf;
}

// All threads; every thread returns the loss. Starts after a barrier that made beta visible.
__device__ double selection_loss(const SearchState& s, double hh, const double* beta)
{
    for (int l = s.tid; l < s.na; l += kSearchThreads) {
        double row = 0.0;
#pragma unroll 8
        for (int m = 0; m < s.na; ++m) row = __dadd_rn(row, __dmul_rn(s.G[l * s.Lp + m], beta[m]));
        s.tmp[l] = row;
    }
    __syncthreads();
    double quad = 0.0, lin = 0.0;
#pragma unroll 8
    for (int l = 0; l < s.na; ++l) {
        quad = __dadd_rn(quad, __dmul_rn(beta[l], s.tmp[l]));
        lin = __dadd_rn(lin, __dmul_rn(s.b[l], beta[l]));
    }
    __syncthreads();
    return __ddiv_rn(__dadd_rn(__dadd_rn(hh, -__dmul_rn(2.0, lin)), quad), s.nrows);
}

// Eq. 9 on the support S (ns atoms): G_SS gamma = b_S by Cholesky in A; gamma lands in s.tmp[0..ns). Right-looking: an
// entry gets its subtractions column by column, which is the order of the sequential inner products. Thread = row.
__device__ bool refit_gamma(const SearchState& s, int ns)
{
    const int Lp = s.Lp, i = s.tid;
    double* A = s.A;
    double* y = s.tmp;
    double* Ai = A + i * (i + 1) / 2;                         // row i
    if (i < ns) {
        for (int j = 0; j <= i; ++j) Ai[j] = s.G[s.S[i] * Lp + s.S[j]];
        y[i] = s.b[s.S[i]];
    }
    __syncthreads();
    for (int j = 0; j < ns; ++j) {
        const double djj = A[j * (j + 1) / 2 + j];
        if (!(djj > 0.0)) return false;                       // the same value in every thread
        const double dj = __dsqrt_rn(djj);
        double lij = 0.0;
        if (i > j && i < ns) {
            lij = __ddiv_rn(Ai[j], dj);
            Ai[j] = lij;
        }
        __syncthreads();
        if (i == j) Ai[j] = dj;
        if (i > j && i < ns) {
#pragma unroll 4
            for (int q = j + 1; q <= i; ++q) Ai[q] = __dadd_rn(Ai[q], -__dmul_rn(lij, A[q * (q + 1) / 2 + j]));
        }
        __syncthreads();
    }
    for (int j = 0; j < ns; ++j) {                            // forward, column by column
        if (i == j) y[j] = __ddiv_rn(y[j], Ai[j]);
        __syncthreads();
        if (i > j && i < ns) y[i] = __dadd_rn(y[i], -__dmul_rn(Ai[j], y[j]));
        __syncthreads();
    }
    for (int j = ns - 1; j >= 0; --j) {                       // backward: the sum runs upwards, so only its products are parallel
        if (i > j && i < ns) s.prod[i] = __dmul_rn(Ai[j], y[i]);
        __syncthreads();
        if (i == j) {
            double v = y[j];
#pragma unroll 8
            for (int q = j + 1; q < ns; ++q) v = __dadd_rn(v, -s.prod[q]);
            y[j] = __ddiv_rn(v, Ai[j]);
        }
        __syncthreads();
    }
    return true;
}

__global__ void __launch_bounds__(kSearchThreads, 1)
selection_search_kernel(const __grid_constant__ SearchParams p)
{
    extern __shared__ __align__(16) double ssm[];
    __shared__ int sCount[kSearchWarps], sAt[kSearchWarps];   // this block's nodes: coefficients that are not zero, and where they are
    __shared__ int sTree[kSearchCtas * kSearchWarps][2];      // the same of all blocks
    cg::cluster_group cluster = cg::this_cluster();
    const int cta = (int)cluster.block_rank(), warps = (int)cluster.num_blocks() * kSearchWarps;
    const int levels = 31 - __clz(warps);                     // of a round's tree: a warp per node
    SearchState s;
    const int L = p.L;
    s.L8 = search_l8(L); s.Lp = s.L8 + 1; s.tid = threadIdx.x; s.lane = threadIdx.x & 31; s.nrows = p.nrows;
    s.na = L;
    double* v = ssm;
    s.diag = v; v += s.L8; s.rcp = v; v += s.L8; s.rcl = v; v += s.L8; s.frz = v; v += s.L8;
    s.b = v; v += s.L8; s.beta = v; v += s.L8; s.r = v; v += s.L8; s.best = v; v += s.L8;
    s.gtot = v; v += s.L8; s.tmp = v; v += s.L8; s.prod = v; v += s.L8;
    s.sub = v; v += s.L8;
    s.solve = v; v += kSearchWarps * 2 * s.L8;
    s.G = v; v += s.L8 * s.Lp;
    s.A = v; v += L * (L + 1) / 2;
    s.S = reinterpret_cast<int*>(v);
    s.orig = s.S + s.L8;
    const int tid = s.tid;
    for (int e = tid; e < L * L; e += kSearchThreads) s.G[(e / L) * s.Lp + (e % L)] = p.G[e];
    for (int l = tid; l < L; l += kSearchThreads) { s.b[l] = p.b[l]; s.beta[l] = 1.0; s.gtot[l] = 1.0; s.orig[l] = l; }
    __syncthreads();
    prepare_active(s);
    const double hh = *p.hh;
    double alpha_t = 1.0, lambda = p.lambda0;
    int step = 0;
    bool failed = false;
    auto copy = [&](double* dst, const double* src) {          // ends in a barrier
        for (int l = tid; l < s.na; l += kSearchThreads) dst[l] = src[l];
        __syncthreads();
    };
    while (alpha_t > p.alpha + 1e-12 && step < p.max_steps && !failed) {
        const double alpha_next = fmax(p.alpha, __dadd_rn(1.0, -__dmul_rn((double)(step + 1), p.dalpha)));
        const double target = __dmul_rn(alpha_next, (double)L), band = __dmul_rn(p.eps, (double)L);
        int solves = 0;
        int nnz = count_nonzero(s, s.beta);
        double lam_hi = lambda;
        // doubling
        while ((double)nnz > target) {
            residuals(s, s.beta);
            if (tid < 32) {
                const double* now = lasso_cd(s, lambda, s.beta, p.tol, p.max_sweeps);
                for (int l = s.lane; l < s.na; l += 32) s.beta[l] = now[l];
            }
            __syncthreads();
            ++solves;
            nnz = count_nonzero(s, s.beta);
            lam_hi = lambda;
            lambda = __dmul_rn(2.0, lambda);
            // Atoms whose G[l][l] is not positive keep beta = 1 at every lambda. When more of them than the target are
            // left, no lambda is large enough: the search has failed once doubling no longer makes it larger.
            if ((double)nnz > target && !(lambda > lam_hi)) { failed = true; break; }
        }
        if (failed) break;
        copy(s.best, s.beta);
        int best_nnz = nnz;
        double best_lam = lam_hi;
        // bisection inside the last doubling step: warp w of the cluster solves node w + 1 of the tree of mid points below
        // [left, right] (children of node i: 2 i, the lower half, and 2 i + 1), then every block walks down that tree. The walk ends
        // where the coefficients that all of it started from are replaced.
        double left = __dmul_rn(0.5, lam_hi), right = lam_hi;
        int it = 0;
        bool stale = true;                                     // s.r does not belong to s.best
        while (fabs(__dadd_rn(target, -(double)nnz)) > band && it < p.max_bisect) {
            if (stale) residuals(s, s.best);
            stale = false;
            const int node = cta * kSearchWarps + (tid >> 5) + 1, level = 31 - __clz(node);
            if (level < levels && it + level < p.max_bisect) {
                double lo = left, hi = right, mid = __dmul_rn(0.5, __dadd_rn(lo, hi));
                for (int u = level - 1; u >= 0; --u) {
                    if ((node >> u) & 1) lo = mid;
                    else hi = mid;
                    mid = __dmul_rn(0.5, __dadd_rn(lo, hi));
                }
                const double* now = lasso_cd(s, mid, s.best, p.tol, p.max_sweeps);
                const int count = count_nonzero(s, now);
                if (s.lane == 0) { sCount[tid >> 5] = count; sAt[tid >> 5] = (int)(now - s.solve); }
            }
            cluster.sync();
            if (tid < warps) {
                sTree[tid][0] = cluster.map_shared_rank(sCount, tid / kSearchWarps)[tid % kSearchWarps];
                sTree[tid][1] = cluster.map_shared_rank(sAt, tid / kSearchWarps)[tid % kSearchWarps];
            }
            __syncthreads();
            int at = 1;
            while (at < (1 << levels) && fabs(__dadd_rn(target, -(double)nnz)) > band && it < p.max_bisect) {
                const double mid = __dmul_rn(0.5, __dadd_rn(left, right));
                ++solves;
                ++it;
                nnz = sTree[at - 1][0];
                const bool in_band_feasible = fabs(__dadd_rn(target, -(double)nnz)) <= band && (double)nnz <= target;
                if (((double)nnz <= target && nnz > best_nnz) || in_band_feasible) {
                    const double* from = cluster.map_shared_rank(s.solve, (at - 1) / kSearchWarps) + sTree[at - 1][1];
                    for (int l = tid; l < s.na; l += kSearchThreads) s.best[l] = from[l];
                    best_nnz = nnz;
                    best_lam = mid;
                    stale = true;
                }
                if ((double)nnz < target) { right = mid; at = 2 * at; }
                else if ((double)nnz > target) { left = mid; at = 2 * at + 1; }
                else break;                                    // the interval stays: the same mid point again
                if (stale) break;
            }
            cluster.sync();                                    // everybody has read the nodes
        }
        copy(s.beta, s.best);
        lambda = best_lam;
        const double loss_beta = selection_loss(s, hh, s.beta);
        // W-step: re-fit on the support
        int ns = 0;
        for (int l0 = 0; l0 < s.na; l0 += 32) {               // every warp counts, warp 0 writes the list
            const int l = l0 + s.lane;
            const unsigned m = __ballot_sync(0xffffffffu, l < s.na && s.beta[l] != 0.0);
            if (tid < 32 && ((m >> s.lane) & 1u)) s.S[ns + __popc(m & ((1u << s.lane) - 1u))] = l;
            ns += __popc(m);
        }
        __syncthreads();
        if (ns == 0 || !refit_gamma(s, ns)) { failed = true; break; }
        // gamma (in tmp[0..ns)) folded into G, b and the running product; the kept atoms become the active set, moved
        // together eight rows at a time (row i comes from row S[i] >= i, so a batch never overwrites a later one's rows)
        for (int i0 = 0; i0 < ns; i0 += 8) {
            double row[8];
            if (tid < ns) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (i0 + u < ns) row[u] = __dmul_rn(__dmul_rn(s.tmp[i0 + u], s.G[s.S[i0 + u] * s.Lp + s.S[tid]]), s.tmp[tid]);
            }
            __syncthreads();
            if (tid < ns) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (i0 + u < ns) s.G[(i0 + u) * s.Lp + tid] = row[u];
            }
            __syncthreads();
        }
        double bi = 0.0, gi = 0.0;
        int oi = 0;
        if (tid < ns) {
            bi = __dmul_rn(s.tmp[tid], s.b[s.S[tid]]);
            gi = __dmul_rn(s.gtot[s.S[tid]], s.tmp[tid]);
            oi = s.orig[s.S[tid]];
        }
        __syncthreads();
        if (tid < ns) { s.b[tid] = bi; s.gtot[tid] = gi; s.orig[tid] = oi; s.beta[tid] = 1.0; }
        s.na = ns;
        __syncthreads();
        prepare_active(s);
        const double loss_gamma = selection_loss(s, hh, s.beta);
        if (p.trace && cta == 0 && tid == 0) {
            double* tr = p.trace + (size_t)step * 6;
            tr[0] = alpha_next; tr[1] = best_lam; tr[2] = (double)ns; tr[3] = loss_beta; tr[4] = loss_gamma; tr[5] = (double)solves;
        }
        alpha_t = alpha_next;
        ++step;
    }
    if (cta != 0) return;
    if (!failed)
        for (int l = tid; l < s.na; l += kSearchThreads) { p.idx_out[l] = (uint8_t)s.orig[l]; p.gamma_out[l] = (float)s.gtot[l]; }
    if (tid == 0) {
        *p.count_out = failed ? -1 : s.na;
        if (p.steps_out) *p.steps_out = step;
    }
}

} // namespace

int selection_gram_slots() { return sm_count(); }

size_t selection_gram_slot_bytes(int D)
{
    const int Dp = (D + 15) / 16 * 16;
    return (size_t)(Dp * Dp + Dp + 8) * sizeof(double);
}

cudaError_t launch_selection_gram(const float* lr, const void* coef, int coef_dtype, const float* dict, const float* target,
                                  const int64_t* samples, int64_t nsamples, double* G, double* b, double* hh, const Problem& pb,
                                  double* slots, int nslots, cudaStream_t st)
{
    GramParams p{};
    p.lr = lr; p.coef = coef; p.coef_f16 = coef_dtype == SR_F16 ? 1 : 0; p.dict = dict; p.target = target; p.samples = samples;
    p.count = samples ? nsamples : (int64_t)pb.n * pb.H * pb.W;
    p.pb = pb;
    p.slots = slots;
    p.Dp = (pb.D + 15) / 16 * 16;
    const int T = pb.D > 32 ? 8 : 4, kk = pb.k * pb.k;       // few atoms: smaller blocks, so that there are enough of them
    p.nb = (pb.D + T - 1) / T;
    p.nblk = p.nb * (p.nb + 1) / 2;
    p.nw = (pb.k - 1 + pb.r - 1) / pb.r + 4;
    const int Dz = p.nb * T;
    auto up4 = [](int v) { return (v + 3) & ~3; };
    p.groups = kGramRank / p.nblk;
    if (p.groups > kGramMaxGroups) p.groups = kGramMaxGroups;
    // No fp32 sum has more terms than 32 pixels give (grey images got 80 of them for a while: up to 20 units in the last place
    // instead of 8).
    const int terms = 32 * pb.c < kGramRows ? 32 * pb.c : kGramRows;
    int64_t most = sm_count();                               // thread blocks
    if (most > nslots) most = nslots;
    // as many pixels per chunk as give at most 96 rows, keep to the terms and fit, but not fewer chunks than blocks as long as
    // a chunk has more than eight pixels (1160 pixels, D = 16: 19.4 us against 27.2 with 80); the divisors of 160 let a producer thread keep its
    // pixel
    int floats = 0;
    for (int px : {80, 40, 32, 20, 16, 8, 4}) {
        if (px * pb.c > kGramRows || px * pb.c > terms * p.groups) continue;
        if (px > 8 && (p.count + px - 1) / px < most) continue;
        p.px = px;
        p.rows = px * pb.c;
        p.off_acc = up4(kk * Dz);
        p.off_set = p.off_acc + up4(2 * (T * T * p.nblk + Dz + 1));
        p.off_z = up4(kk * (((p.rows + 7) & ~7) + 4));
        p.off_h = p.off_z + p.rows * Dz;
        p.off_win = p.off_h + 2 * kGramRows;
        p.off_phi = p.off_win + up4(p.rows * p.nw * p.nw);
        p.set_floats = p.off_phi + up4(pb.D * p.px + (pb.D >> 3) * 4);
        floats = p.off_set + 2 * p.set_floats;
        if ((size_t)floats * sizeof(float) <= (size_t)kGramSmemMax) break;
        floats = 0;
    }
    if (floats == 0) return cudaErrorNotSupported;
    const size_t smem = (size_t)floats * sizeof(float);
    auto magic = [](int d) { return (uint32_t)((0x100000000ull + d - 1) / d); };
    p.px_magic = magic(p.px); p.nw_magic = magic(p.nw); p.nb_magic = magic(p.nb); p.r_magic = magic(pb.r); p.rows_magic = magic(p.rows);
    const int rows_per_group = (p.rows + p.groups - 1) / p.groups;
    p.flush_every = terms / rows_per_group > 1 ? terms / rows_per_group : 1;
    const int64_t chunks = (p.count + p.px - 1) / p.px;
    int64_t ctas = most;
    if (ctas > chunks) ctas = chunks;
    if (ctas < 1) ctas = 1;
    cudaError_t e;
    switch (pb.k) {
    case 1: e = launch_gram_k<1>(p, T, (int)ctas, smem, st); break;
    case 3: e = launch_gram_k<3>(p, T, (int)ctas, smem, st); break;
    case 5: e = launch_gram_k<5>(p, T, (int)ctas, smem, st); break;
    case 7: e = launch_gram_k<7>(p, T, (int)ctas, smem, st); break;
    case 9: e = launch_gram_k<9>(p, T, (int)ctas, smem, st); break;
    default: return cudaErrorNotSupported;
    }
    if (e != cudaSuccess) return e;
    selection_gram_reduce_kernel<<<(pb.D * pb.D + pb.D + 1 + 31) / 32, dim3(32, kReduceLanes), 0, st>>>(slots, (int)ctas, p.Dp, pb.D, G, b, hh);
    count_launches(1);
    return cudaGetLastError();
}

// ---- the Gram kernel without caller scratch --------------------------------------------------------------------------
//
// Some users of this library may not allocate device memory at the point where they want the Gram statistics: a
// video pipeline that sizes all of its buffers once at start-up and runs under a fixed memory budget afterwards, a
// plug-in inside a host application that owns the allocator, a service whose steady state must not call cudaMalloc
// because that call synchronises the whole device and can fail long after start-up. For them the per-CTA fp64 slots of
// selection_gram_kernel live in the array below instead of in memory the caller passes: kStaticGramSlots slots for at
// most kStaticGramMaxD atoms, 32 x (80 x 80 + 80 + 8) doubles = 1 660 928 bytes that every device which loads the
// library holds until the process exits. The array is shared by all calls and keeps what the last call left in it:
// every CTA overwrites what is read of its slot, once, at its end, and two calls whose kernels could run at the same time
// (two streams, two host threads) must not both use this entry point, or one would read the other's slots.
constexpr int kStaticGramSlots = 32;
constexpr int kStaticGramMaxD = 80;
static __device__ __align__(256) double g_gram_static_slots[kStaticGramSlots * (kStaticGramMaxD * kStaticGramMaxD + kStaticGramMaxD + 8)];

int selection_gram_static_max_atoms() { return kStaticGramMaxD; }

// Device address of the array above on the current device. In host code the array's name only stands for the symbol;
// the address a kernel can use comes from cudaGetSymbolAddress, looked up once per device while that device is current.
static double* static_gram_slots()
{
    static double* cache[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!cache[dev]) {
        double* ptr = nullptr;
        if (cudaGetSymbolAddress((void**)&ptr, g_gram_static_slots) != cudaSuccess) return nullptr;
        cache[dev] = ptr;
    }
    return cache[dev];
}

cudaError_t launch_selection_gram_static(const float* lr, const void* coef, int coef_dtype, const float* dict, const float* target,
                                         const int64_t* samples, int64_t nsamples, double* G, double* b, double* hh, const Problem& pb,
                                         cudaStream_t st)
{
    if (pb.D > kStaticGramMaxD) return cudaErrorInvalidValue;
    double* slots = static_gram_slots();
    if (!slots) return cudaErrorUnknown;
    return launch_selection_gram(lr, coef, coef_dtype, dict, target, samples, nsamples, G, b, hh, pb, slots, kStaticGramSlots, st);
}

size_t selection_search_scratch_bytes(int L) { return (size_t)L * L * sizeof(double); }

cudaError_t launch_selection_search(const double* G, const double* b, const double* hh, double nrows, int L, const sr_search_opts& o,
                                    uint8_t* idx_out, float* gamma_out, int* count_out, double* trace, int* steps_out, cudaStream_t st)
{
    if (L > kMaxSearchL) return cudaErrorNotSupported;
    SearchParams p{};
    p.G = G; p.b = b; p.hh = hh; p.L = L; p.nrows = nrows;
    p.alpha = o.alpha; p.dalpha = o.delta_alpha; p.eps = o.eps; p.lambda0 = o.lambda0; p.tol = o.tol;
    p.max_sweeps = o.max_sweeps; p.max_bisect = o.max_bisect; p.max_steps = o.max_steps;
    p.idx_out = idx_out; p.gamma_out = gamma_out; p.count_out = count_out; p.trace = trace; p.steps_out = steps_out;
    constexpr auto bytes = [](int l) {
        const size_t l8 = search_l8(l);
        return (12 * l8 + kSearchWarps * 2 * l8 + l8 * (l8 + 1) + (size_t)l * (l + 1) / 2) * sizeof(double) + 2 * l8 * sizeof(int);
    };
    static bool configured[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(selection_search_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kMaxSearchL));
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    cudaLaunchAttribute shape{};
    shape.id = cudaLaunchAttributeClusterDimension;
    shape.val.clusterDim.y = shape.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kSearchThreads);
    cfg.dynamicSmemBytes = bytes(L);
    cfg.stream = st;
    cfg.attrs = &shape;
    cfg.numAttrs = 1;
    for (int ctas = kSearchCtas;; ctas /= 2) {
        shape.val.clusterDim.x = ctas;
        cfg.gridDim = dim3(ctas);
        int fit = 0;
        if (ctas == 1 || (cudaOccupancyMaxActiveClusters(&fit, selection_search_kernel, &cfg) == cudaSuccess && fit > 0)) break;
        (void)cudaGetLastError();                            // (a shape that cannot run leaves nothing behind)
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, selection_search_kernel, p);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

} // namespace sr
