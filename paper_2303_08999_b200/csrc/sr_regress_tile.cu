// Dense and global-subset regression with fp32 coefficients on the fp32 FMA pipe, register-tiled:
//   out[c][i] = sum_j (sum_l w_l Phi_l[i] dict_l[j]) B_{i,c}[j]
// A warp owns 128 pixels of a row, a thread four neighbouring ones: it keeps their filters in registers, and a dictionary
// row read from shared memory (16-byte broadcasts) serves all four. Coefficients travel through a ring of DEPTH planes'
// row pieces per warp (asynchronous copies, 16 bytes where rows are aligned, else 4). With 7 x 7 and 9 x 9 atoms the taps
// are split over NS warps that share the pixels, and their partial results are added at the end through shared memory.
// The up-sampled tile is built after the filters, out of an LR window that travels meanwhile. Neither F nor U reaches
// memory.
//
// Bound: the FMA pipe (D k^2 + c k^2 multiply-adds per pixel). The thread-per-pixel kernel reads a whole dictionary row
// per pixel and atom and is held by the shared-memory pipe at a quarter of that rate. 180 x 320 x3, D = 72, k = 5:
// 118 -> 69 us (27 at the FMA pipe's rate); 540 x 960 x4: 1885 -> 784 us. Where the rest goes: up-sampling, set-up and
// filtering are a third of the instructions, and 12 warps per SM (168 registers) do not hide every load.
// With aligned rows a lane copies the sixteen bytes it reads itself, from a running address where the planes follow one another: no
// warp barrier, and no table of planes to make and wait for before the first copy (180 x 320 x3, D = 72: 5 x 5 63.9 -> 62.0 us, 3 x 3
// 37.4 -> 34.5, 7 x 7 124.5 -> 116.3; with the table still made 63.1, 35.6 and 119.4, and 9 x 9 with few atoms slower than before).
// Measured on the first shape and dropped: coefficients prefetched into registers (PF atoms ahead share the warp's few
// load scoreboards: 78-124 us); tiles of 32 columns x 4 rows per thread (DRAM rows of 128 bytes, 83 us); 16 warps per SM
// (spills, 128 us); scalar multiply-adds (84 us); the taps of 5 x 5 over two or three warps (77-115 us).
#include <math.h>
#include <type_traits>

#include "sr_regress_tile.cuh"
#include "sr_tile_upsample.cuh"

namespace sr {

namespace {

using namespace tile;

struct TileParams {
    const float* lr;
    const float* coef;
    const float* dict;
    void* out;
    const uint8_t* idx;   // atom ids of a subset, or nullptr
    const float* gamma;   // its weights, or nullptr
    Geom g;
    int natoms;
    int planes;           // planes per frame in the coefficient tensor
    int gather;           // 1: the subset's planes are planes idx[q] of the full tensor
    int out_vec;          // 1: fp32 output whose rows take 16-byte stores
    int off_u, off_v, off_l, off_red, off_ring;   // shared-memory offsets in floats
};

// 4- and 16-byte asynchronous copies that read `bytes` of the source and zero the rest
__device__ __forceinline__ void cp4(uint32_t dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int PX = 4;                                    // pixels per thread
constexpr int kStageBytes = 512;                         // a ring slot: 128 pixels

template <int K> __host__ __device__ constexpr int dict_pitch() { return (K * K / 4) * 4 + 4; }   // the 16-byte units, the last tap, zeros

// K: atom side; NS: warps that share the taps; GPC: such groups (rows) per block; CTAS: blocks per SM; VEC: 16-byte copies; GATHER:
// planes by table (always without VEC), else one after the other
template <int K, int NS, int GPC, int CTAS, int DEPTH, bool VEC, bool GATHER>
__global__ void __launch_bounds__(32 * NS * GPC, CTAS) regress_tile_kernel(const __grid_constant__ TileParams p)
{
    constexpr int kk = K * K, P = (K - 1) / 2, UNITS = kk / 4, U = UNITS / NS, PITCH = dict_pitch<K>();
    constexpr int NT = 32 * NS * GPC, UW = tile_uw(P), UW4 = UW / 4, STAGE = kStageBytes;
    constexpr int NU = (PX + K - 1 + 3) / 4;                 // 16-byte loads that cover a thread's four patches in a U row
    static_assert(U * NS == UNITS, "the parts are equal");
    extern __shared__ __align__(16) float smem[];
    __shared__ float wpad[kMaxScale][12];
    const Geom& g = p.g;
    const Problem& pb = g.pb;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int part = warp % NS, grp = warp / NS;
    float* sD = smem;                                        // [natoms][PITCH]
    int64_t* sOff = reinterpret_cast<int64_t*>(smem + p.natoms * PITCH);   // [natoms]: first element of the atom's plane
    float* sU = smem + p.off_u;                              // [C][uh][UW]
    float* sV = smem + p.off_v;                              // [C][uh][tcols]
    float* sL = smem + p.off_l;                              // [C * trows][tcols]
    float* sRed = smem + p.off_red;                          // [C][GPC][NS - 1][PX][32]
    uint8_t* ring = reinterpret_cast<uint8_t*>(smem + p.off_ring) + warp * (DEPTH * STAGE);
    const int C = pb.c, H = pb.H, W = pb.W, natoms = p.natoms;
    const int64_t HW = (int64_t)H * W;

    // ---- set-up
    LrWindow w;
    decode_tile(g, blockIdx.x, w.f, w.y0, w.x0, w.rows);
    lr_window_of_tile<P>(g, w);
    if constexpr (GATHER) {
        for (int l = tid; l < natoms; l += NT) {
            const int plane = p.gather ? min((int)__ldg(p.idx + l), pb.D - 1) : l;
            sOff[l] = ((int64_t)w.f * p.planes + plane) * HW;
        }
    }
    for (int i = tid; i < (p.off_red - p.off_v) / 4; i += NT) reinterpret_cast<float4*>(sV)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (GATHER) __syncthreads();
    // this lane's copies of atom l's piece of the row into slot l mod DEPTH; every call commits one group
    const int row = min(w.y0 + grp, H - 1), x = w.x0 + PX * lane;
    const float* row0 = p.coef + (int64_t)row * W + w.x0;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    const float* mine = row0 + (x < W ? PX * lane : 0) + (GATHER ? 0 : (int64_t)w.f * p.planes * HW);   // VEC: this lane's pixels
    const uint32_t mine_bytes = x < W ? 16u : 0u, mine_s = ring_s + 16 * lane;
    auto fetch = [&](int l, uint32_t slot) {
        if (l < natoms) {
            if constexpr (VEC) {
                cp16(mine_s + slot, GATHER ? mine + sOff[l] : mine, mine_bytes);
                if (!GATHER) mine += HW;
            } else {
                const float* src = row0 + sOff[l];
                const uint32_t dst = ring_s + slot;
#pragma unroll
                for (int i = 0; i < PX; ++i) {
                    const int c = lane + 32 * i;
                    const bool in = w.x0 + c < W;
                    cp4(dst + 4 * c, src + (in ? c : 0), in ? 4u : 0u);
                }
            }
        }
        cp_commit();
    };
#pragma unroll
    for (int u = 0; u < DEPTH - 1; ++u) fetch(u, (uint32_t)(u * STAGE));
    fill_wpad(pb, wpad, tid, NT);
    for (int i = tid; i < natoms * PITCH; i += NT) {
        const int l = i / PITCH, j = i - l * PITCH;
        float v = 0.f;
        if (j < kk) {
            const int a = p.idx ? min((int)__ldg(p.idx + l), pb.D - 1) : l;
            v = __ldg(p.dict + (int64_t)a * kk + j) * (p.gamma ? __ldg(p.gamma + l) : 1.f);
        }
        sD[i] = v;
    }
    __syncthreads();
    prefetch_lr_window_of(g, p.lr, w, sL, tid, NT);          // joins the next group

    // ---- the filters of this thread's pixels: taps 4 U part .. 4 U part + 4 U - 1, and the last tap in the last part
    float2 F[PX][2 * U > 0 ? 2 * U : 1];
    float Fl[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        Fl[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 2 * U; ++j) F[i][j] = make_float2(0.f, 0.f);
    }
    const float* dl = sD + part * (4 * U);
    const int last = part == NS - 1 ? 4 * UNITS - part * (4 * U) : 4 * UNITS + 1 - part * (4 * U);   // the last tap, or a zero
    uint32_t slot = 0, free_slot = (DEPTH - 1) * STAGE;
#pragma unroll 2
    for (int l = 0; l < natoms; ++l, dl += PITCH) {
        cp_wait<DEPTH - 2>();
        // every lane's part of the piece has landed; the slot read last is free (VEC: a lane reads what it copied itself)
        if (!VEC) __syncwarp();
        const float4 v4 = *reinterpret_cast<const float4*>(ring + slot + 16 * lane);
        const float v[PX] = {v4.x, v4.y, v4.z, v4.w};
        fetch(l + DEPTH - 1, free_slot);
        free_slot = slot;
        slot = slot + STAGE == DEPTH * STAGE ? 0 : slot + STAGE;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const float4 d = *reinterpret_cast<const float4*>(dl + 4 * q);
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                F[i][2 * q] = __ffma2_rn(make_float2(d.x, d.y), make_float2(v[i], v[i]), F[i][2 * q]);
                F[i][2 * q + 1] = __ffma2_rn(make_float2(d.z, d.w), make_float2(v[i], v[i]), F[i][2 * q + 1]);
            }
        }
        const float d = dl[last];
#pragma unroll
        for (int i = 0; i < PX; ++i) Fl[i] = fmaf(d, v[i], Fl[i]);
    }

    // ---- the up-sampled tile
    cp_wait<0>();
    __syncthreads();
    {
        const int uh = w.rows + 2 * P, tc4 = g.tcols >> 2;
        const int v_lanes = NT / tc4, v_lane = fast_div(tid, tc4, g.tc4_magic);
        if (v_lane < v_lanes) vertical_pass(g, w, uh, P, sL, sV, (tid - v_lane * tc4) * 4, v_lane, v_lanes);
        __syncthreads();
        constexpr int kHLanes = NT / UW4;
        const int h_lane = tid / UW4;
        if (h_lane < kHLanes) horizontal_pass<P>(g, wpad, w, uh, sV, sU, tid - h_lane * UW4, h_lane, kHLanes);
        __syncthreads();
    }

    // ---- applied: pixel i, tap (a, b) reads row grp + a, column 4 lane + i + b
    const bool clamp01 = (pb.flags & SR_CLAMP01) != 0;
#pragma unroll 1
    for (int c = 0; c < C; ++c) {
        const float* u0 = sU + (c * g.uh + grp) * UW + PX * lane;
        float acc[PX];
#pragma unroll
        for (int i = 0; i < PX; ++i) acc[i] = 0.f;
        auto apply = [&](auto part_c) {
            constexpr int PART = decltype(part_c)::value, T0 = 4 * U * PART, T1 = T0 + 4 * U;
#pragma unroll
            for (int a = 0; a < K; ++a) {
                if ((a * K < T1 && (a + 1) * K > T0) || (PART == NS - 1 && a == K - 1)) {   // this part has taps of patch row a
                    float u[4 * NU];
#pragma unroll
                    for (int n = 0; n < NU; ++n) *reinterpret_cast<float4*>(u + 4 * n) = *reinterpret_cast<const float4*>(u0 + a * UW + 4 * n);
#pragma unroll
                    for (int b = 0; b < K; ++b) {
                        const int t = a * K + b, j = t - T0;
                        if (PART == NS - 1 && t == kk - 1) {
#pragma unroll
                            for (int i = 0; i < PX; ++i) acc[i] = fmaf(Fl[i], u[i + b], acc[i]);
                        } else if (t >= T0 && t < T1) {
#pragma unroll
                            for (int i = 0; i < PX; ++i) acc[i] = fmaf((j & 1) ? F[i][j >> 1].y : F[i][j >> 1].x, u[i + b], acc[i]);
                        }
                    }
                }
            }
        };
        if constexpr (NS == 1) apply(std::integral_constant<int, 0>{});
        else {
            if (part == 0) apply(std::integral_constant<int, 0>{});
            if (part == 1) apply(std::integral_constant<int, 1>{});
            if constexpr (NS > 2) { if (part == 2) apply(std::integral_constant<int, 2>{}); }
            if constexpr (NS > 3) { if (part == 3) apply(std::integral_constant<int, 3>{}); }
            // the parts' sums meet in the last part's warp, in order
            float* red = sRed + ((c * GPC + grp) * (NS - 1)) * PX * 32 + lane;
            if (part < NS - 1) {
#pragma unroll
                for (int i = 0; i < PX; ++i) red[(part * PX + i) * 32] = acc[i];
            }
            asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(32 * NS) : "memory");
            if (part == NS - 1) {
#pragma unroll
                for (int q = 0; q < NS - 1; ++q)
#pragma unroll
                    for (int i = 0; i < PX; ++i) acc[i] += red[(q * PX + i) * 32];
            }
        }
        if (part == NS - 1 && grp < w.rows) {
            const int64_t o = ((int64_t)w.f * C + c) * HW + (int64_t)row * W + x;
            float v[PX];
#pragma unroll
            for (int i = 0; i < PX; ++i) v[i] = clamp01 ? fminf(fmaxf(acc[i], 0.f), 1.f) : acc[i];
            if (VEC && p.out_vec) {
                if (x < W) *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + o) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int i = 0; i < PX; ++i)
                    if (x + i < W) store_out(reinterpret_cast<float*>(p.out), o + i, v[i], pb.flags);
            }
        }
    }
}

constexpr int kTileSmemMax = 200 * 1024;

// Warps that share the taps, groups (rows) per block, blocks per SM and ring slots for atoms of side K.
template <int K> struct Shape;
template <> struct Shape<1> { static constexpr int NS = 1, GPC = 4, CTAS = 6, DEPTH = 8; };
template <> struct Shape<3> { static constexpr int NS = 1, GPC = 4, CTAS = 4, DEPTH = 12; };
template <> struct Shape<5> { static constexpr int NS = 1, GPC = 4, CTAS = 3, DEPTH = 8; };
template <> struct Shape<7> { static constexpr int NS = 2, GPC = 2, CTAS = 3, DEPTH = 8; };
template <> struct Shape<9> { static constexpr int NS = 4, GPC = 2, CTAS = 2, DEPTH = 8; };

// Fills the tile geometry and the shared-memory offsets for natoms atoms; returns bytes.
template <int K> size_t plan_tile(TileParams& prm, const Problem& pb)
{
    using S = Shape<K>;
    plan_geom(prm.g, pb, S::GPC, prm.lr);
    const Geom& g = prm.g;
    auto up4 = [](int v) { return (v + 3) & ~3; };
    prm.off_u = up4(prm.natoms * dict_pitch<K>() + 2 * prm.natoms);
    prm.off_v = prm.off_u + up4(pb.c * g.uh * tile_uw((K - 1) / 2));
    prm.off_l = prm.off_v + up4(pb.c * g.uh * g.tcols);
    prm.off_red = prm.off_l + up4(pb.c * g.trows * g.tcols + 8);
    prm.off_ring = prm.off_red + pb.c * PX * S::GPC * (S::NS - 1) * 32;
    return (size_t)prm.off_ring * sizeof(float) + (size_t)S::NS * S::GPC * S::DEPTH * kStageBytes;
}

template <int K, bool VEC, bool GATHER>
cudaError_t launch_v(TileParams& prm, const Problem& pb, cudaStream_t st)
{
    using S = Shape<K>;
    const size_t smem = plan_tile<K>(prm, pb);
    if (smem > (size_t)kTileSmemMax) return cudaErrorNotSupported;
    auto kern = regress_tile_kernel<K, S::NS, S::GPC, S::CTAS, S::DEPTH, VEC, GATHER>;
    static bool configured[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemMax);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    kern<<<(unsigned)prm.g.num_tiles, 32 * S::NS * S::GPC, smem, st>>>(prm);
    count_launches(1);
    return cudaGetLastError();
}

template <int K>
cudaError_t launch_t(TileParams& prm, const Problem& pb, cudaStream_t st)
{
    if ((pb.W & 3) == 0 && (reinterpret_cast<uintptr_t>(prm.coef) & 15) == 0)
        return prm.gather ? launch_v<K, true, true>(prm, pb, st) : launch_v<K, true, false>(prm, pb, st);
    return launch_v<K, false, true>(prm, pb, st);
}

// The kernel's expected time, us: a launch, the dictionary by atom, what an SM's tiles cost together and what each turn of the
// blocks that fit an SM costs, either of them as such, by atom, by channel and by channel over the scale. Fitted to 1045 of the
// frames that regress_general_us is fitted to (standard deviation 6 to 8 %; 1 x 1 12 %).
struct Cost { float launch, dict, tile, tile_atom, tile_channel, tile_lr, turn, turn_atom, turn_channel, turn_lr; };
template <int K> float tile_us(int natoms, const Problem& pb, const Cost& c)
{
    TileParams prm{};
    prm.natoms = natoms;
    const size_t smem = plan_tile<K>(prm, pb);
    if (smem > (size_t)kTileSmemMax) return INFINITY;
    const int sms = sm_count(), fit = (int)(228 * 1024 / (smem + 1536));      // (1536: the kernel's own arrays and the system's kilobyte)
    const int blocks = fit < 1 ? 1 : (fit < Shape<K>::CTAS ? fit : Shape<K>::CTAS);
    const float tiles = (float)prm.g.num_tiles / sms, turns = (float)((prm.g.num_tiles + sms * blocks - 1) / (sms * blocks));
    return c.launch + c.dict * natoms + tiles * (c.tile + c.tile_atom * natoms + pb.c * (c.tile_channel + c.tile_lr / pb.r)) +
           turns * (c.turn + c.turn_atom * natoms + pb.c * (c.turn_channel + c.turn_lr / pb.r));
}

float estimate(const Problem& pb, int natoms)
{
    switch (pb.k) {
    case 1: return tile_us<1>(natoms, pb, {2.85f, 0.006f, 0.30f, 0.027f, 0.03f, 0.11f, 0.f, 0.043f, 0.14f, 0.54f});
    case 3: return tile_us<3>(natoms, pb, {2.79f, 0.017f, 0.47f, 0.023f, 0.06f, 0.10f, 0.35f, 0.083f, 0.14f, 0.78f});
    case 5: return tile_us<5>(natoms, pb, {2.54f, 0.085f, 0.41f, 0.062f, 0.14f, 0.07f, 0.98f, 0.057f, 0.05f, 1.02f});
    case 7: return tile_us<7>(natoms, pb, {3.12f, 0.081f, 0.66f, 0.035f, 0.19f, 0.f, 0.f, 0.168f, 0.f, 1.27f});
    default: return tile_us<9>(natoms, pb, {3.38f, 0.020f, 1.29f, 0.077f, 0.29f, 0.f, 0.f, 0.236f, 0.21f, 1.00f});
    }
}

} // namespace

bool regress_tile_supported(int mode, int coef_dtype, const Problem& pb)
{
    if ((mode != kModeDense && mode != kModeGlobal) || coef_dtype != SR_F32 || pb.c > 4 || (pb.flags & SR_LUMA_ONLY)) return false;
    // Tiles of 512 pixels and three blocks per SM only pay once they fill the chip; the thread-per-pixel kernel is faster
    // on less than about one block per SM (64 x 64, x2, 5 x 5: 14.6 us against 18.4).
    if ((int64_t)pb.n * pb.H * pb.W < (int64_t)sm_count() * 512) return false;
    // A tile works on 128 columns however narrow the frame, the other kernel on 32 x 8 pixels, and large tables leave one block
    // on an SM: by expected times (on the 1045 frames 31 lose more than 6 % against the better kernel, 35 % at most; batches of 32
    // columns would take 1.6 to 3.4 times as long here, full tiles take 0.5 to 0.8 of the other's time).
    return estimate(pb, mode == kModeGlobal ? pb.s : pb.D) < regress_general_us(mode, SR_F32, pb);
}

cudaError_t launch_regress_tile(int mode, const float* lr, const void* coef, const uint8_t* idx, const float* gamma, const float* dict,
                                float* out, const Problem& pb, cudaStream_t st)
{
    TileParams prm{};
    prm.lr = lr; prm.coef = static_cast<const float*>(coef); prm.dict = dict; prm.out = out;
    if (mode == kModeGlobal) {
        prm.idx = idx; prm.gamma = gamma;
        prm.natoms = pb.s;
        prm.gather = (pb.flags & SR_COEF_COMPACT) ? 0 : 1;
        prm.planes = prm.gather ? pb.D : pb.s;
    } else {
        prm.natoms = prm.planes = pb.D;
    }
    prm.out_vec = (pb.W & 3) == 0 && !(pb.flags & (SR_OUT_F16 | SR_OUT_U8)) && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    switch (pb.k) {
    case 1: return launch_t<1>(prm, pb, st);
    case 3: return launch_t<3>(prm, pb, st);
    case 5: return launch_t<5>(prm, pb, st);
    case 7: return launch_t<7>(prm, pb, st);
    case 9: return launch_t<9>(prm, pb, st);
    default: return cudaErrorNotSupported;
    }
}

} // namespace sr
