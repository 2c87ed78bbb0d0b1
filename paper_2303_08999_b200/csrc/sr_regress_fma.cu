// General regression kernel on the fp32 FMA pipe: every shape, fp32 or binary16 coefficients, all modes.
// It is the path for small and narrow frames and the fallback for shapes and alignments the others do not take; dense and
// global-subset frames large enough go to the register-tiled kernel (fp32) or the row kernel (binary16), those that one block per
// multiprocessor covers to the split kernel (launch_regress_fma).
//
// One thread per HR pixel, 32 x 8 pixel tiles. Per pixel: assemble the filter F = Phi_i D in registers
// (dictionary rows broadcast from shared memory), then y_c = F . B_c against an up-sampled tile with a
// halo of p = (k-1)/2 that lives only in shared memory. Neither F nor the patch matrix B reaches HBM.
#include "sr_pick.cuh"
#include "sr_regress_rows.cuh"
#include "sr_regress_split.cuh"
#include "sr_regress_tile.cuh"
#include <type_traits>

namespace sr {

namespace {

// Selection inside the call with lists beyond pick_top's sixteen: a kernel of its own, so that those networks' registers do not
// cost it blocks (1 x 1 and 3 x 3 atoms: 64 registers instead of 48).
constexpr int kModeFusedLong = 5;

constexpr int TX = 32, TY = 8, CCHUNK = 4;

template <int K> struct KK { static constexpr int value = K * K, padded = (K * K + 3) & ~3; };

// (magnitude, lower index first) as one ordered integer; unique per atom.
__device__ __forceinline__ long long select_key(uint32_t mag, int l) { return ((long long)mag << 8) | (long long)(255 - l); }

template <int K, typename CoefT, int MODE>
__global__ void __launch_bounds__(TX * TY)
regress_fma_kernel(const float* __restrict__ lr, const CoefT* __restrict__ coef, const uint8_t* __restrict__ idx,
                   const float* __restrict__ gamma, const float* __restrict__ dict, float* __restrict__ out,
                   const __grid_constant__ Problem pb)
{
    constexpr int kk = KK<K>::value, kkp = KK<K>::padded, P = (K - 1) / 2;
    constexpr int UW = TX + 2 * P, UH = TY + 2 * P;
    extern __shared__ __align__(16) float smem[];
    float* sdict = smem;                         // [D][kkp]
    float* sU = smem + (size_t)pb.D * kkp;       // [CCHUNK][UH][UW]

    const int tid = threadIdx.y * TX + threadIdx.x;
    const int X = blockIdx.x * TX + threadIdx.x, Y = blockIdx.y * TY + threadIdx.y;
    const int f = blockIdx.z;
    const int H = pb.H, W = pb.W, D = pb.D, s = pb.s;
    const int64_t HW = (int64_t)H * W;
    const bool valid = X < W && Y < H;
    const int64_t pix = (int64_t)min(Y, H - 1) * W + min(X, W - 1);

    for (int i = tid; i < D * kkp; i += TX * TY) {
        const int l = i / kkp, j = i - l * kkp;
        sdict[i] = j < kk ? __ldg(dict + (int64_t)l * kk + j) : 0.f;
    }
    __syncthreads();

    // ---- stage 3: F = sum_q weight_q * dict[atom_q]
    float F[kkp];
#pragma unroll
    for (int j = 0; j < kkp; ++j) F[j] = 0.f;
    auto accumulate = [&](int atom, float wgt) {
        const float4* row = reinterpret_cast<const float4*>(sdict + atom * kkp);
#pragma unroll
        for (int j4 = 0; j4 < kkp / 4; ++j4) {
            const float4 dv = row[j4];
            F[4 * j4 + 0] = fmaf(wgt, dv.x, F[4 * j4 + 0]);
            F[4 * j4 + 1] = fmaf(wgt, dv.y, F[4 * j4 + 1]);
            F[4 * j4 + 2] = fmaf(wgt, dv.z, F[4 * j4 + 2]);
            F[4 * j4 + 3] = fmaf(wgt, dv.w, F[4 * j4 + 3]);
        }
    };
    if (MODE == kModeDense) {
        const CoefT* cp = coef + (int64_t)f * D * HW + pix;
        // loads in flight: small frames wait for nothing else; 9 x 9 filters leave no registers for twelve (53 binary16 frames
        // above 20 000 pixels: 2 % slower than with four on average, 14 % at most)
        constexpr int AHEAD = K == 9 ? 4 : 12;
        int l0 = 0;
        for (; l0 + AHEAD <= D; l0 += AHEAD) {
            float v[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) v[u] = load_coef(cp, (int64_t)(l0 + u) * HW);
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) accumulate(l0 + u, v[u]);
        }
        for (; l0 < D; ++l0) accumulate(l0, load_coef(cp, (int64_t)l0 * HW));
    } else if (MODE == kModeIdx) {
        for (int q = 0; q < s; ++q) {
            const int a = min((int)__ldg(idx + ((int64_t)f * s + q) * HW + pix), D - 1);
            accumulate(a, load_coef(coef, ((int64_t)f * D + a) * HW + pix));
        }
    } else if (MODE == kModeCompact) {
        for (int q = 0; q < s; ++q) {
            const int a = min((int)__ldg(idx + ((int64_t)f * s + q) * HW + pix), D - 1);
            accumulate(a, load_coef(coef, ((int64_t)f * s + q) * HW + pix));
        }
    } else if (MODE == kModeGlobal) {
        const bool compact = (pb.flags & SR_COEF_COMPACT) != 0;
        for (int q = 0; q < s; ++q) {
            const int a = min((int)__ldg(idx + q), D - 1);
            const float g = gamma ? __ldg(gamma + q) : 1.f;
            const int64_t plane = compact ? ((int64_t)f * s + q) : ((int64_t)f * D + a);
            accumulate(a, g * load_coef(coef, plane * HW + pix));
        }
    } else if (MODE == kModeFusedSelect) { // s <= 16: the list in registers, its values fetched again (from L1 or L2 by now); fp32 748 x 660 x3: 2809 -> 868 us
        const CoefT* cp = coef + (int64_t)f * D * HW + pix;
        uint32_t list[4] = {0, 0, 0, 0};                     // a byte per atom
        auto pick = [&](auto tag) {
            constexpr int S = decltype(tag)::value;
            int atom[S];
            pick_top<S, CoefT>(cp, HW, D, s, atom);
#pragma unroll
            for (int i = 0; i < S; ++i) list[i / 4] |= (uint32_t)atom[i] << (8 * (i % 4));
        };
        if (s == 1) pick(std::integral_constant<int, 1>{});
        else if (s == 2) pick(std::integral_constant<int, 2>{});
        else if (s <= 4) pick(std::integral_constant<int, 4>{});
        else if (s <= 8) pick(std::integral_constant<int, 8>{});
        else pick(std::integral_constant<int, 16>{});
        for (int q = 0; q < s; ++q) {
            const int a = (int)(list[0] & 255u);
            list[0] = __funnelshift_r(list[0], list[1], 8);
            list[1] = __funnelshift_r(list[1], list[2], 8);
            list[2] = __funnelshift_r(list[2], list[3], 8);
            list[3] >>= 8;
            accumulate(a, load_coef(cp, (int64_t)a * HW));
        }
    } else { // kModeFusedLong: repeated scan for the next-largest key; any s, any D
        const CoefT* cp = coef + (int64_t)f * D * HW + pix;
        long long prev = 0x7FFFFFFFFFFFFFFFll;
        for (int q = 0; q < s; ++q) {
            long long best = -1;
            for (int l = 0; l < D; ++l) {
                const long long key = select_key(mag_bits(__ldg(cp + (int64_t)l * HW)), l);
                if (key < prev && key > best) best = key;
            }
            prev = best;
            const int a = 255 - (int)(best & 255);
            accumulate(a, load_coef(cp, (int64_t)a * HW));
        }
    }

    // ---- stages 1 + 4, CCHUNK channels at a time
    const int Y0 = blockIdx.y * TY - P, X0 = blockIdx.x * TX - P;
    for (int c0 = 0; c0 < pb.c; c0 += CCHUNK) {
        const int nc = min(CCHUNK, pb.c - c0);
        __syncthreads();
        for (int i = tid; i < nc * UH * UW; i += TX * TY) {
            const int ch = i / (UH * UW), rem = i - ch * (UH * UW);
            const int uy = rem / UW, ux = rem - uy * UW;
            const float* plane = lr + ((int64_t)f * pb.c + c0 + ch) * pb.h * pb.w;
            sU[i] = bicubic_point(plane, pb.h, pb.w, pb.r, pb.ph, clampi(Y0 + uy, 0, H - 1), clampi(X0 + ux, 0, W - 1));
        }
        __syncthreads();
        if (pb.flags & SR_LUMA_ONLY) {
            // c = 3 (checked by the caller): the fourth slot takes the luma of the tile, the filter runs on it once,
            // and every channel moves by the same amount, so the chroma differences stay those of stage 1.
            float* sY = sU + 3 * UH * UW;
            for (int i = tid; i < UH * UW; i += TX * TY)
                sY[i] = fmaf(0.299f, sU[i], fmaf(0.587f, sU[UH * UW + i], 0.114f * sU[2 * UH * UW + i]));
            __syncthreads();
            const float* u = sY + threadIdx.y * UW + threadIdx.x;
            float acc = 0.f;
#pragma unroll
            for (int a = 0; a < K; ++a)
#pragma unroll
                for (int b = 0; b < K; ++b) acc = fmaf(F[a * K + b], u[a * UW + b], acc);
            const float shift = acc - u[P * UW + P];
            for (int ch = 0; ch < 3; ++ch) {
                float v = sU[ch * UH * UW + (threadIdx.y + P) * UW + threadIdx.x + P] + shift;
                if (pb.flags & SR_CLAMP01) v = fminf(fmaxf(v, 0.f), 1.f);
                if (valid) store_out(out, ((int64_t)f * 3 + ch) * HW + pix, v, pb.flags);
            }
            break;
        }
        for (int ch = 0; ch < nc; ++ch) {
            const float* u = sU + ch * UH * UW + threadIdx.y * UW + threadIdx.x;
            float acc = 0.f;
#pragma unroll
            for (int a = 0; a < K; ++a)
#pragma unroll
                for (int b = 0; b < K; ++b) acc = fmaf(F[a * K + b], u[a * UW + b], acc);
            if (pb.flags & SR_CLAMP01) acc = fminf(fmaxf(acc, 0.f), 1.f);
            if (valid) store_out(out, ((int64_t)f * pb.c + c0 + ch) * HW + pix, acc, pb.flags);
        }
    }
}

template <int K, typename CoefT, int MODE>
cudaError_t launch_t(const float* lr, const void* coef, const uint8_t* idx, const float* gamma, const float* dict,
                     float* out, const Problem& pb, cudaStream_t st)
{
    constexpr int P = (K - 1) / 2;
    const size_t smem = ((size_t)pb.D * KK<K>::padded + (size_t)CCHUNK * (TY + 2 * P) * (TX + 2 * P)) * sizeof(float);
    auto kern = regress_fma_kernel<K, CoefT, MODE>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((pb.W + TX - 1) / TX, (pb.H + TY - 1) / TY, pb.n), block(TX, TY);
    if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
    kern<<<grid, block, smem, st>>>(lr, (const CoefT*)coef, idx, gamma, dict, out, pb);
    count_launches(1);
    return cudaGetLastError();
}

template <int K, typename CoefT>
cudaError_t launch_m(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma,
                     const float* dict, float* out, const Problem& pb, cudaStream_t st)
{
    switch (mode) {
    case kModeDense: return launch_t<K, CoefT, kModeDense>(lr, coef, idx, gamma, dict, out, pb, st);
    case kModeIdx: return launch_t<K, CoefT, kModeIdx>(lr, coef, idx, gamma, dict, out, pb, st);
    case kModeCompact: return launch_t<K, CoefT, kModeCompact>(lr, coef, idx, gamma, dict, out, pb, st);
    case kModeGlobal: return launch_t<K, CoefT, kModeGlobal>(lr, coef, idx, gamma, dict, out, pb, st);
    default: return pb.s <= 16 ? launch_t<K, CoefT, kModeFusedSelect>(lr, coef, idx, gamma, dict, out, pb, st)
                               : launch_t<K, CoefT, kModeFusedLong>(lr, coef, idx, gamma, dict, out, pb, st);
    }
}

template <typename CoefT>
cudaError_t launch_k(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma,
                     const float* dict, float* out, const Problem& pb, cudaStream_t st)
{
    switch (pb.k) {
    case 1: return launch_m<1, CoefT>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    case 3: return launch_m<3, CoefT>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    case 5: return launch_m<5, CoefT>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    case 7: return launch_m<7, CoefT>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    default: return launch_m<9, CoefT>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    }
}

} // namespace

// A launch, the dictionary by atom, and per block of 32 x 8 pixels that an SM works off: by atom and by channel. Subsets fetch
// plane by plane where dense launches keep twelve loads in flight. Fitted to 3100 frames of 33 000 to nine million pixels, 8 to 4000
// columns, scales 1 to 4, 1 to 256 atoms (standard deviation 5 to 10 %).
float regress_general_us(int mode, int coef_dtype, const Problem& pb)
{
    struct Cost { float launch, dict, dict_subset, atom, atom_subset, channel; };
    constexpr Cost f16[3] = {{3.72f, 0.024f, 0.038f, 0.027f, 0.048f, 0.61f}, {4.06f, 0.044f, 0.048f, 0.060f, 0.099f, 0.84f},
                             {4.24f, 0.075f, 0.056f, 0.116f, 0.218f, 1.13f}};                       // 3 x 3, 5 x 5, 7 x 7
    constexpr Cost f32[5] = {{3.49f, 0.006f, 0.026f, 0.018f, 0.036f, 0.40f}, {3.61f, 0.026f, 0.036f, 0.028f, 0.049f, 0.62f},
                             {4.21f, 0.034f, 0.f, 0.065f, 0.109f, 0.82f}, {5.24f, 0.052f, 0.f, 0.121f, 0.245f, 1.06f},
                             {4.02f, 0.f, 0.172f, 0.279f, 0.257f, 1.97f}};                          // 1 x 1 to 9 x 9
    const int i = pb.k / 2;
    const Cost& c = coef_dtype == SR_F16 ? f16[i < 1 ? 0 : (i > 3 ? 2 : i - 1)] : f32[i > 4 ? 4 : i];
    const bool subset = mode == kModeGlobal;
    const int natoms = subset ? pb.s : pb.D;
    const float blocks = (float)((double)pb.n * ((pb.W + TX - 1) / TX) * ((pb.H + TY - 1) / TY) / sm_count());
    return c.launch + (subset ? c.dict_subset : c.dict) * natoms + blocks * ((subset ? c.atom_subset : c.atom) * natoms + c.channel * pb.c);
}

cudaError_t launch_regress_fma(int mode, const float* lr, const void* coef, int coef_dtype, const uint8_t* idx,
                               const float* gamma, const float* dict, float* out, const Problem& pb, cudaStream_t st, bool split)
{
    if (split && regress_split_pays(mode, coef_dtype, pb))
        return launch_regress_split(mode, lr, coef, coef_dtype, idx, gamma, dict, out, pb, st);
    if (regress_tile_supported(mode, coef_dtype, pb)) return launch_regress_tile(mode, lr, coef, idx, gamma, dict, out, pb, st);
    if (regress_rows_form(mode, coef_dtype, pb) && regress_rows_pay(mode, pb)) return launch_regress_rows(mode, lr, coef, idx, gamma, dict, out, pb, st);
    if (coef_dtype == SR_F16) return launch_k<__half>(mode, lr, coef, idx, gamma, dict, out, pb, st);
    return launch_k<float>(mode, lr, coef, idx, gamma, dict, out, pb, st);
}

} // namespace sr
