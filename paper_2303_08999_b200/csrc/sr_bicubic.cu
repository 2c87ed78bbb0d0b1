// Stage 1 alone: bicubic up-sampling of every LR plane (Keys a = -0.75, half-pixel centres, edge clamp).
// A thread produces a BS x BS block of HR pixels from one LR window, separably (bicubic_block_kernel): BS = 4 at scales
// 1, 2 and 4, BS = 6 or 3 at scale 3, BS = r above. The direct 4 x 4 form (bicubic_kernel: one thread, four consecutive
// pixels of a row) remains for scales the block kernel is not instantiated for.
// Vector stores when the row pitch allows it; the LR taps come through the read-only cache.
#include "sr_common.cuh"

namespace sr {

__global__ void __launch_bounds__(256) bicubic_kernel(const float* __restrict__ lr, float* __restrict__ hr,
                                                      const __grid_constant__ Problem pb)
{
    const int W = pb.W, H = pb.H;
    const int groups = (W + 3) >> 2;
    const int64_t total = (int64_t)pb.n * pb.c * H * groups;
    const bool vec = (W & 3) == 0 && ((reinterpret_cast<uintptr_t>(hr) & 15) == 0);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t % groups);
        const int64_t row = t / groups;          // plane * H + Y
        const int Y = (int)(row % H);
        const int64_t plane = row / H;
        const float* src = lr + plane * (int64_t)pb.h * pb.w;
        const int X0 = g * 4;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = (X0 + i < W) ? bicubic_point(src, pb.h, pb.w, pb.r, pb.ph, Y, X0 + i) : 0.f;
        float* dst = hr + row * (int64_t)W + X0;
        if (vec) {
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (X0 + i < W) dst[i] = v[i];
        }
    }
}

// First LR tap of phase p at scale r, relative to X / r (the same integer arithmetic as the host's phase table).
__host__ __device__ constexpr int phase_base(int p, int r)
{
    const int num = 2 * p + 1 - r;
    return (num >= 0 ? num / (2 * r) : -((-num + 2 * r - 1) / (2 * r))) - 1;
}

// One thread produces a column of `run` blocks of BS x BS HR pixels, BS a multiple of the scale. A block starts on a
// multiple of the scale, so every pixel's phase and the offset of its taps inside the block's LR window are compile-time
// constants: a horizontal pass gives BS values per window row and a vertical pass the BS^2 outputs. The next block down
// starts BS / R LR rows further on and shares the other NWIN - BS / R filtered rows with this one, so after the first block
// a thread only loads and filters BS / R new rows (scale 4: 5 loads and 80 multiply-adds per 16 pixels instead of 25
// and 144).
// Bound: HBM / L2 writes in the limit; at 1080p the instructions of about one wave of threads. 270 x 480 x4, device time:
// 11.0 -> 7.0 us, four frames 1080 x 1920 x2: 142 -> 94 us (before: a block per thread, 64-bit index divisions, every
// window row loaded and filtered for every block).
template <int R, int BS>
__global__ void __launch_bounds__(128) bicubic_block_kernel(const float* __restrict__ lr, float* __restrict__ hr,
                                                            const __grid_constant__ Problem pb, int run, unsigned flat)
{
    static_assert(BS % R == 0, "a block starts on a multiple of the scale");
    constexpr int B0 = phase_base(0, R), STEP = BS / R;
    constexpr int NWIN = (BS - 1) / R + phase_base((BS - 1) % R, R) - B0 + 4;    // window side: last pixel's first tap + 4
    constexpr int VEC = BS % 4 == 0 ? 4 : (BS % 2 == 0 ? 2 : 1);                 // floats per store
    const int W = pb.W, H = pb.H, w = pb.w, h = pb.h;
    const unsigned bw = (unsigned)(W + BS - 1) / BS, bh = (unsigned)(H + BS - 1) / BS, runs = (bh + run - 1) / run;
    // a block's threads share a plane, or (flat: threads per plane) thread after thread goes to plane after plane
    const int64_t planes = (int64_t)pb.n * pb.c;
    unsigned t = blockIdx.x * 128u + threadIdx.x;
    int64_t plane = blockIdx.y, next = gridDim.y;
    if (flat) {
        plane = t / flat;
        t -= (unsigned)plane * flat;
        next = planes;
    }
    const unsigned ry = t / bw, bx = t - ry * bw;
    if (ry >= runs) return;
    const bool vec = VEC > 1 && (W % VEC) == 0 && ((reinterpret_cast<uintptr_t>(hr) & (4 * VEC - 1)) == 0) && BS * (int)bx + BS <= W;
    const int col0 = STEP * (int)bx + B0;
    int cx[NWIN];
#pragma unroll
    for (int c = 0; c < NWIN; ++c) cx[c] = clampi(col0 + c, 0, w - 1);
    for (; plane < planes; plane += next) {
        const float* src = lr + plane * (int64_t)h * w;
        float T[NWIN][BS];                                   // horizontal pass of the window's rows
        auto filter_row = [&](int j, int y) {                // LR row y (clamped) into window row j
            const float* row = src + clampi(y, 0, h - 1) * w;
            float L[NWIN];
#pragma unroll
            for (int c = 0; c < NWIN; ++c) L[c] = __ldg(row + cx[c]);
#pragma unroll
            for (int i = 0; i < BS; ++i) {
                const int off = i / R + phase_base(i % R, R) - B0;   // compile-time after unrolling
                float a = pb.ph.w[i % R][0] * L[off];
                a = fmaf(pb.ph.w[i % R][1], L[off + 1], a);
                a = fmaf(pb.ph.w[i % R][2], L[off + 2], a);
                a = fmaf(pb.ph.w[i % R][3], L[off + 3], a);
                T[j][i] = a;
            }
        };
        const int by0 = (int)ry * run, by1 = min(by0 + run, (int)bh);
        int y = STEP * by0 + B0;
#pragma unroll
        for (int j = STEP; j < NWIN; ++j) filter_row(j, y + j - STEP);     // all but the rows the first turn brings
        float* dst = hr + (plane * H + BS * by0) * (int64_t)W + BS * (int)bx;
        for (int by = by0; by < by1; ++by, y += STEP, dst += (int64_t)BS * W) {
            // the window moves down: STEP rows leave, STEP new ones come
#pragma unroll
            for (int j = 0; j + STEP < NWIN; ++j)
#pragma unroll
                for (int i = 0; i < BS; ++i) T[j][i] = T[j + STEP][i];
#pragma unroll
            for (int j = NWIN - STEP; j < NWIN; ++j) filter_row(j, y + j);
#pragma unroll
            for (int k = 0; k < BS; ++k) {
                if (BS * by + k >= H) break;
                const int off = k / R + phase_base(k % R, R) - B0;
                float v[BS];
#pragma unroll
                for (int i = 0; i < BS; ++i) {
                    float a = pb.ph.w[k % R][0] * T[off][i];
                    a = fmaf(pb.ph.w[k % R][1], T[off + 1][i], a);
                    a = fmaf(pb.ph.w[k % R][2], T[off + 2][i], a);
                    a = fmaf(pb.ph.w[k % R][3], T[off + 3][i], a);
                    v[i] = a;
                }
                float* o = dst + (int64_t)k * W;
                if (vec) {
#pragma unroll
                    for (int i = 0; i < BS; i += VEC) {
                        if constexpr (VEC == 4) *reinterpret_cast<float4*>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                        else *reinterpret_cast<float2*>(o + i) = make_float2(v[i], v[i + 1]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < BS; ++i)
                        if (BS * (int)bx + i < W) o[i] = v[i];
                }
            }
        }
    }
}

template <int R, int BS>
static cudaError_t launch_block(const float* lr, float* hr, const Problem& pb, cudaStream_t st)
{
    const int64_t bw = (pb.W + BS - 1) / BS, bh = (pb.H + BS - 1) / BS, planes = (int64_t)pb.n * pb.c;
    // blocks per thread: as many as leave about twenty warps per SM (270 x 480 x4, threads per SM asked for: 256 8.0 us,
    // 640 7.0, 1024 7.4, a block per thread 9.1), up to 4 (540 x 960 x4: 1 / 2 / 4 / 8 blocks 30.5 / 23.2 / 20.2 / 22.5 us;
    // 705 x 1261 x3: 42.5 / 29.8 / 25.9 / 28.1; four frames 1080 x 1920 x2: 127 / 98 / 91 / 94)
    int64_t run = bw * bh * planes / ((int64_t)sm_count() * 640);
    // one where a frame is less than four blocks wide: the lanes of a warp then take blocks one below the other
    run = run < 1 || bw < 4 ? 1 : (run > 4 ? 4 : run);
    const int64_t threads = bw * ((bh + run - 1) / run);
    // planes of a few blocks of threads leave too much of the last one idle: their threads follow one another (batches of small
    // frames and frames up to 16 columns wide: without this and the rule above up to 2.4 times the time of a block per thread)
    const bool flat = planes > 1 && threads < 1024 && threads * planes < ((int64_t)1 << 31);
    const dim3 grid((unsigned)(((flat ? threads * planes : threads) + 127) / 128), flat ? 1u : (unsigned)(planes < 65535 ? planes : 65535));
    bicubic_block_kernel<R, BS><<<grid, 128, 0, st>>>(lr, hr, pb, (int)run, flat ? (unsigned)threads : 0u);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_bicubic(const float* lr, float* hr, const Problem& pb, cudaStream_t st)
{
    switch (pb.r) {
    case 1: return launch_block<1, 4>(lr, hr, pb, st);
    case 2: return launch_block<2, 4>(lr, hr, pb, st);
    case 3:
        // 6 x 6 blocks store float2 but need an even width; rows of odd width and large frames take 3 x 3 blocks, whose
        // smaller windows leave more warps (6 x 6 / 3 x 3, us: 180 x 320 3.9 / 4.6, 360 x 640 8.4 / 8.7, two planes
        // 872 x 1736 30.0 / 28.5; odd widths 333 x 501 8.9 / 6.8, 705 x 1261 39.3 / 25.9)
        if ((pb.W & 1) != 0 || (int64_t)pb.n * pb.c * pb.h * pb.w > 1000000) return launch_block<3, 3>(lr, hr, pb, st);
        return launch_block<3, 6>(lr, hr, pb, st);
    case 4: return launch_block<4, 4>(lr, hr, pb, st);
    case 5: return launch_block<5, 5>(lr, hr, pb, st);
    case 6: return launch_block<6, 6>(lr, hr, pb, st);
    default: break;
    }
    const int64_t total = (int64_t)pb.n * pb.c * pb.H * ((pb.W + 3) >> 2);
    int64_t blocks = (total + 255) / 256;
    const int64_t cap = (int64_t)sm_count() * 8 * 4;
    if (blocks > cap) blocks = cap;
    bicubic_kernel<<<(unsigned)blocks, 256, 0, st>>>(lr, hr, pb);
    count_launches(1);
    return cudaGetLastError();
}

} // namespace sr
