// Dense and global-subset regression of small frames, fp32 or binary16 coefficients, any width.
//
// A frame of some ten thousand pixels gives a thread per pixel a warp or two per scheduler, and each of them waits for one trip
// to memory per dozen atoms, then for the dictionary, then for the LR image: the time is a sum of latencies. Here a pixel has NS threads,
// one per warp of a row's group, with every NS-th atom each. A thread asks for its coefficients first (up to twenty, eighty atoms
// of a pixel), then for its entries of the dictionary and the LR taps of its values of the up-sampled tile, and waits once for all
// of them. Each warp applies its part of the filter to the patch, and the parts' sums meet in shared memory, a channel per warp.
// One block of 32 x 4 pixels per SM. 64 x 64 x2, D = 72, 5 x 5, fp32: 13.0 -> 8.6 us of device time. Bound: launch and one trip to
// memory (3.7 us), a channel's part of the tile and of the filtering (0.5 us), 0.045 us an atom of 5 x 5 (issue slots of sixteen
// warps). Tiles of 32 x 2 with 256 threads took 9.4 us there; the up-sampled tile in two passes through shared memory, after its LR
// window, 8.8.

#include "sr_regress_split.cuh"
#include "sr_tile_upsample.cuh"

namespace sr {

namespace {

using namespace tile;

constexpr int TWD = 32, NT = 512, kWarps = NT / 32;
constexpr int NS = 4;                                    // threads of a pixel
constexpr int ROWS = kWarps / NS;                        // tile height
constexpr int kAhead = 20;                               // coefficients a thread has in flight

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__half v) { return __half2float(v); }

template <int K> __host__ __device__ constexpr int dict_pitch() { return (K * K + 3) & ~3; }

struct SplitParams {
    const float* lr;
    const void* coef;
    const float* dict;
    float* out;
    const uint8_t* idx;   // atom ids of a subset, or nullptr
    const float* gamma;   // its weights, or nullptr
    Geom g;
    int natoms;
    int planes;           // planes per frame in the coefficient tensor
    int gather;           // 1: the subset's planes are planes idx[q] of the full tensor
    int off_u, off_red;   // shared-memory offsets in floats
};

template <int K, typename CoefT>
__global__ void __launch_bounds__(NT, 1) regress_split_kernel(const __grid_constant__ SplitParams p)
{
    constexpr int kk = K * K, P = (K - 1) / 2, PITCH = dict_pitch<K>(), UW = TWD + 2 * P, UH = ROWS + 2 * P;
    extern __shared__ __align__(16) float smem[];
    const Geom& g = p.g;
    const Problem& pb = g.pb;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, part = warp % NS, row = warp / NS;
    float* sD = smem;                                        // [natoms][PITCH]
    float* sU = smem + p.off_u;                              // [C][UH][UW]
    float* sRed = smem + p.off_red;                          // [C][NS][ROWS * 32]
    const int C = pb.c, natoms = p.natoms;
    const int64_t HW = (int64_t)pb.H * pb.W;

    int f, y0, x0, rows;
    decode_tile(g, blockIdx.x, f, y0, x0, rows);
    const int X = x0 + lane, Y = y0 + row;
    const int64_t pix = (int64_t)min(Y, pb.H - 1) * pb.W + min(X, pb.W - 1);
    const CoefT* cp = static_cast<const CoefT*>(p.coef) + (int64_t)f * p.planes * HW + pix;
    CoefT v[kAhead];
    auto fetch = [&](int l0) {                               // (beyond the atoms: the last one again, not used)
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int l = min(l0 + u * NS, natoms - 1);
            v[u] = __ldg(cp + (int64_t)(p.gather ? min((int)__ldg(p.idx + l), pb.D - 1) : l) * HW);
        }
    };
    fetch(part);
    auto dict_entry = [&](int i) {
        const int l = i / PITCH, j = i - l * PITCH;
        if (i >= natoms * PITCH || j >= kk) return 0.f;
        const int a = p.idx ? min((int)__ldg(p.idx + l), pb.D - 1) : l;
        return __ldg(p.dict + (int64_t)a * kk + j) * (p.gamma ? __ldg(p.gamma + l) : 1.f);
    };
    constexpr int kDict = 4;                                 // dictionary entries a thread has in flight
    float dv[kDict];
#pragma unroll
    for (int u = 0; u < kDict; ++u) dv[u] = dict_entry(tid + u * NT);

    // ---- the up-sampled tile, sixteen taps a value: they travel with the loads above, two passes through shared memory would follow them
#pragma unroll 2
    for (int i = tid; i < C * UH * UW; i += NT) {
        const int ch = i / (UH * UW), rem = i - ch * (UH * UW), uy = rem / UW, ux = rem - uy * UW;
        int py, px;
        const int ty = first_tap(g, clampi(y0 - P + uy, 0, pb.H - 1), py), tx = first_tap(g, clampi(x0 - P + ux, 0, pb.W - 1), px);
        const float* plane = p.lr + ((int64_t)f * C + ch) * pb.h * pb.w;
        float v = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float* src = plane + (int64_t)clampi(ty + a, 0, pb.h - 1) * pb.w;
            float t = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) t = fmaf(pb.ph.w[px][b], __ldg(src + clampi(tx + b, 0, pb.w - 1)), t);
            v = fmaf(pb.ph.w[py][a], t, v);
        }
        sU[i] = v;
    }
#pragma unroll
    for (int u = 0; u < kDict; ++u)
        if (tid + u * NT < natoms * PITCH) sD[tid + u * NT] = dv[u];
#pragma unroll 4
    for (int i = tid + kDict * NT; i < natoms * PITCH; i += NT) sD[i] = dict_entry(i);
    __syncthreads();

    // ---- this warp's part of the filters
    float2 F[PITCH / 2];
#pragma unroll
    for (int j = 0; j < PITCH / 2; ++j) F[j] = make_float2(0.f, 0.f);
    for (int l0 = part; l0 < natoms; l0 += kAhead * NS) {
        if (l0 != part) fetch(l0);
        const float* dl = sD + l0 * PITCH;
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (l0 + u * NS < natoms) {
                const float2 phi = make_float2(to_float(v[u]), to_float(v[u]));
#pragma unroll
                for (int q = 0; q < PITCH / 4; ++q) {
                    const float4 d = *reinterpret_cast<const float4*>(dl + u * (NS * PITCH) + 4 * q);
                    F[2 * q] = __ffma2_rn(make_float2(d.x, d.y), phi, F[2 * q]);
                    F[2 * q + 1] = __ffma2_rn(make_float2(d.z, d.w), phi, F[2 * q + 1]);
                }
            }
        }
    }

    // ---- applied; the parts' sums in order
    for (int c = 0; c < C; ++c) {
        const float* u = sU + (c * UH + row) * UW + lane;
        float acc = 0.f;
#pragma unroll
        for (int a = 0; a < K; ++a)
#pragma unroll
            for (int b = 0; b < K; ++b) {
                const int t = a * K + b;
                acc = fmaf((t & 1) ? F[t >> 1].y : F[t >> 1].x, u[a * UW + b], acc);
            }
        sRed[(c * NS + part) * (ROWS * 32) + row * 32 + lane] = acc;
    }
    __syncthreads();
    for (int c = part; c < C; c += NS) {
        const float* r = sRed + c * NS * (ROWS * 32) + row * 32 + lane;
        float acc = r[0];
#pragma unroll
        for (int q = 1; q < NS; ++q) acc += r[q * (ROWS * 32)];
        if (pb.flags & SR_CLAMP01) acc = fminf(fmaxf(acc, 0.f), 1.f);
        if (X < pb.W && Y < pb.H) store_out(p.out, ((int64_t)f * C + c) * HW + pix, acc, pb.flags);
    }
}

constexpr int kSplitSmemMax = 160 * 1024;                // 256 atoms of 9 x 9, four channels: 111 KB

template <int K> size_t plan_split(SplitParams& prm, const Problem& pb)
{
    constexpr int P = (K - 1) / 2;
    plan_geom(prm.g, pb, ROWS, prm.lr, TWD);
    prm.off_u = prm.natoms * dict_pitch<K>();
    prm.off_red = prm.off_u + pb.c * (ROWS + 2 * P) * (TWD + 2 * P);
    return (size_t)(prm.off_red + pb.c * NS * ROWS * 32) * sizeof(float);
}

template <int K, typename CoefT>
cudaError_t launch_t(SplitParams& prm, const Problem& pb, cudaStream_t st)
{
    const size_t smem = plan_split<K>(prm, pb);
    if (smem > (size_t)kSplitSmemMax) return cudaErrorNotSupported;
    auto kern = regress_split_kernel<K, CoefT>;
    static bool configured[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmemMax);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    kern<<<(unsigned)prm.g.num_tiles, NT, smem, st>>>(prm);
    count_launches(1);
    return cudaGetLastError();
}

template <int K>
cudaError_t launch_k(SplitParams& prm, int coef_dtype, const Problem& pb, cudaStream_t st)
{
    return coef_dtype == SR_F16 ? launch_t<K, __half>(prm, pb, st) : launch_t<K, float>(prm, pb, st);
}

} // namespace

// On 408 frames that one block per multiprocessor covers (up to 18 900 pixels; 4 to 200 atoms, subsets among them): 0.80 of the
// time of what served them before, 361 of them faster. Where atoms and channels are few there is nothing to deal out and the
// thread-per-pixel kernel's shorter set-up wins (32 of them: 1.03 to 1.26, one-channel frames of eight atoms and less above all).
// The line, on 512 frames of 1 to 24 atoms and of one to four channels on either side of it: geometric means 0.78 to 0.98 above it,
// 7 x 7 with three channels, 14 atoms 0.95 (12 1.00, 8 1.02), with four, six 0.98 (five 1.01, four 1.04, one 1.05), 3 x 3 with one
// channel, 26 atoms 1.00 (24 1.06). Aligned binary16 frames with much to multiply stay on the tensor cores (96 atoms of 7 x 7 32 x
// 32 x2 14.8 us against 13.7; 128 17.4 against 14.9). A second turn of blocks costs all of the first again: 0.88 of the best other
// time at 14 000 to 19 000 pixels, 1.4 just above.
bool regress_split_pays(int mode, int coef_dtype, const Problem& pb)
{
    if ((mode != kModeDense && mode != kModeGlobal) || pb.c > 4 || (pb.flags & SR_LUMA_ONLY) || pb.k < 3) return false;
    const int64_t tiles = (int64_t)pb.n * ((pb.W + TWD - 1) / TWD) * ((pb.H + ROWS - 1) / ROWS);
    const int natoms = mode == kModeGlobal ? pb.s : pb.D;
    const int least = 32 + (pb.k == 7 && pb.c >= 3 ? 6 : 0) + (pb.k == 3 && pb.c == 1 ? 2 : 0);
    if (tiles > sm_count() || natoms + 8 * pb.c < least) return false;
    return !(coef_dtype == SR_F16 && (pb.W & 7) == 0 && pb.k <= 7 && natoms * pb.k * pb.k > 4000);
}

cudaError_t launch_regress_split(int mode, const float* lr, const void* coef, int coef_dtype, const uint8_t* idx, const float* gamma,
                                 const float* dict, float* out, const Problem& pb, cudaStream_t st)
{
    SplitParams prm{};
    prm.lr = lr; prm.coef = coef; prm.dict = dict; prm.out = out;
    if (mode == kModeGlobal) {
        prm.idx = idx; prm.gamma = gamma;
        prm.natoms = pb.s;
        prm.gather = (pb.flags & SR_COEF_COMPACT) ? 0 : 1;
        prm.planes = prm.gather ? pb.D : pb.s;
    } else {
        prm.natoms = prm.planes = pb.D;
    }
    switch (pb.k) {
    case 3: return launch_k<3>(prm, coef_dtype, pb, st);
    case 5: return launch_k<5>(prm, coef_dtype, pb, st);
    case 7: return launch_k<7>(prm, coef_dtype, pb, st);
    case 9: return launch_k<9>(prm, coef_dtype, pb, st);
    default: return cudaErrorNotSupported;
    }
}

} // namespace sr
