// The ordered kernel's block sums from half the pair terms (7,681 to 32,768 padded ions).
//
// k_forces<128, IPT> sums each target's terms over one block of 128 sources after another, every
// block from zero in ascending source order.  This kernel makes the same block sums, bit for
// bit, and evaluates each unordered pair once: the term c3 (r_j - r_i) is the same number for
// both ions up to its sign.  A warp takes two blocks of targets, one per half-warp, eight
// consecutive targets per lane, and 128 packets of two sources (ion p of each of two blocks).
// The packets pass through a half-warp as a wave, lane l one step behind lane l - 1, so that
// every target meets the sources in ascending order; a packet's own sum travels with it,
// through the lane's eight targets in order and then one lane up, so that every source meets the
// targets in ascending order, and comes out complete at the half-warp's last lane.
//
// blk[b][c][i] (b: source block, c: x, y, z): the block sums, which k_fold_blocks adds up in the
// ordered kernel's slots.  At the two ends of a wave 15 of 143 steps find no packet and read
// one far away, whose terms are exactly zero.
#include <algorithm>

#include "od_device.cuh"

namespace od {

constexpr int WAVE_B = 128;           // ions per block
constexpr int WAVE_TI = 2 * WAVE_B;   // ions per tile (two blocks)
constexpr int WAVE_BT = 64;           // threads per CTA (two independent warps)
constexpr int WAVE_T = 8;             // targets per lane
constexpr int WAVE_LAG = WAVE_B / WAVE_T - 1;
constexpr int WAVE_STEPS = WAVE_B + WAVE_LAG + 1;  // a multiple of four
// The dynamic unit queue taken one warp at a time (a CTA's warps are independent of each other).
__device__ __forceinline__ long long next_warp_unit(unsigned long long* sched)
{
    unsigned long long u = 0;
    if ((threadIdx.x & 31) == 0) u = atomicAdd(sched, 1ull);
    return (long long)__shfl_sync(0xffffffffu, u, 0);
}

__device__ __forceinline__ void leave_warp_queue(unsigned long long* sched)
{
    if ((threadIdx.x & 31) == 0 && atomicAdd(sched + 1, 1ull) == (unsigned long long)gridDim.x * (blockDim.x >> 5) - 1) {
        sched[0] = 0ull;
        sched[1] = 0ull;
    }
}

struct WaveStage {
    f32x2 x[WAVE_STEPS + WAVE_LAG], y[WAVE_STEPS + WAVE_LAG], z[WAVE_STEPS + WAVE_LAG];  // packet p at LAG + p
    f32x2 out[2][3][WAVE_STEPS];  // sums of packet p from each block of targets, at LAG + p
};

// this lane's eight values to consecutive floats at dst (16-byte aligned)
__device__ __forceinline__ void put8(float* dst, const float (&v)[WAVE_T])
{
    reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

__global__ void __launch_bounds__(WAVE_BT, 65536 / (WAVE_BT * 168))
    k_forces_wave(const float4* __restrict__ fpos, ForceArgs F)
{
    __shared__ WaveStage stage[WAVE_BT / 32];
    WaveStage& S = stage[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, hl = lane & 15, half = lane >> 4;
    const int T = F.n_pad / WAVE_TI;
    const long long U = (long long)T * (T + 1) / 2, ld = F.n_pad;
    if (lane <= WAVE_LAG) {
        const f32x2 far = pk2(9.0e4f, 9.0e4f);
        if (lane < WAVE_LAG) S.x[lane] = S.y[lane] = S.z[lane] = far;
        const int q = WAVE_LAG + WAVE_B + lane;
        S.x[q] = S.y[q] = S.z[q] = far;
    }
    for (;;) {
        const long long u = next_warp_unit(F.sched);
        if (u >= U) break;
        int I, J;
        tri_unit(u, T, I, J);
        __syncwarp();  // the previous unit's reads are done
#pragma unroll
        for (int q = 0; q < WAVE_B / 32; ++q) {
            const int p = q * 32 + lane;
            const float4 a = __ldg(fpos + J * WAVE_TI + p), b = __ldg(fpos + J * WAVE_TI + WAVE_B + p);
            S.x[WAVE_LAG + p] = pk2(a.x, b.x);
            S.y[WAVE_LAG + p] = pk2(a.y, b.y);
            S.z[WAVE_LAG + p] = pk2(a.z, b.z);
        }
        const int i0 = I * WAVE_TI + lane * WAVE_T;
        float xi[WAVE_T], yi[WAVE_T], zi[WAVE_T];
        f32x2 ax[WAVE_T], ay[WAVE_T], az[WAVE_T];
#pragma unroll
        for (int k = 0; k < WAVE_T; ++k) {
            const float4 p = __ldg(fpos + i0 + k);
            xi[k] = p.x;
            yi[k] = p.y;
            zi[k] = p.z;
            ax[k] = ay[k] = az[k] = 0ull;
        }
        __syncwarp();
        if (I == J) {
            // the tile itself: its ordered pairs (every lane reads the same packet)
#pragma unroll 4
            for (int t = 0; t < WAVE_B; ++t) {
                const f32x2 xj = S.x[WAVE_LAG + t], yj = S.y[WAVE_LAG + t], zj = S.z[WAVE_LAG + t];
#pragma unroll
                for (int k = 0; k < WAVE_T; ++k) {
                    const f32x2 dx = sub2(xj, pk2(xi[k], xi[k])), dy = sub2(yj, pk2(yi[k], yi[k])),
                                dz = sub2(zj, pk2(zi[k], zi[k]));
                    const f32x2 c3 = pair_c3x2(dx, dy, dz);
                    ax[k] = fma2(c3, dx, ax[k]);
                    ay[k] = fma2(c3, dy, ay[k]);
                    az[k] = fma2(c3, dz, az[k]);
                }
            }
        } else {
            const int first = WAVE_LAG - hl;
            f32x2 bx = 0ull, by = 0ull, bz = 0ull;
#pragma unroll 4
            for (int t = 0; t < WAVE_STEPS; ++t) {
                const f32x2 xj = S.x[first + t], yj = S.y[first + t], zj = S.z[first + t];
#pragma unroll
                for (int k = 0; k < WAVE_T; ++k) {
                    const f32x2 dx = sub2(xj, pk2(xi[k], xi[k])), dy = sub2(yj, pk2(yi[k], yi[k])),
                                dz = sub2(zj, pk2(zi[k], zi[k]));
                    const f32x2 c3 = pair_c3x2(dx, dy, dz);
                    bx = fma2(c3, dx, bx);
                    by = fma2(c3, dy, by);
                    bz = fma2(c3, dz, bz);
                    ax[k] = fma2(c3, dx, ax[k]);
                    ay[k] = fma2(c3, dy, ay[k]);
                    az[k] = fma2(c3, dz, az[k]);
                }
                if (hl == WAVE_LAG) {
                    S.out[half][0][t] = bx;
                    S.out[half][1][t] = by;
                    S.out[half][2][t] = bz;
                }
                bx = __shfl_up_sync(0xffffffffu, bx, 1);
                by = __shfl_up_sync(0xffffffffu, by, 1);
                bz = __shfl_up_sync(0xffffffffu, bz, 1);
                if (hl == 0) bx = by = bz = 0ull;
            }
            __syncwarp();
            // the sources' sums, made with the targets' sign
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float a[4], b[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) upk2(S.out[n][c][WAVE_LAG + 4 * lane + k], a[k], b[k]);
                    float4* dst = reinterpret_cast<float4*>(F.blk + ((2ll * I + n) * 3 + c) * ld + J * WAVE_TI) + lane;
                    dst[0] = make_float4(-a[0], -a[1], -a[2], -a[3]);
                    dst[WAVE_B / 4] = make_float4(-b[0], -b[1], -b[2], -b[3]);
                }
        }
        float* dst = F.blk + (2ll * J) * 3 * ld + i0;
        float a[WAVE_T], b[WAVE_T];
#pragma unroll
        for (int k = 0; k < WAVE_T; ++k) upk2(ax[k], a[k], b[k]);
        put8(dst, a);
        put8(dst + 3 * ld, b);
#pragma unroll
        for (int k = 0; k < WAVE_T; ++k) upk2(ay[k], a[k], b[k]);
        put8(dst + ld, a);
        put8(dst + 4 * ld, b);
#pragma unroll
        for (int k = 0; k < WAVE_T; ++k) upk2(az[k], a[k], b[k]);
        put8(dst + 2 * ld, a);
        put8(dst + 5 * ld, b);
    }
    leave_warp_queue(F.sched);
}

// The ordered kernel's partial slots from the block sums: slot s of tile t is the sum, in block
// order, over the chunks that its block s covers (blockIdx.x = t, blockIdx.y = s).
__global__ void __launch_bounds__(WAVE_TI) k_fold_blocks(float4* __restrict__ part, ForceArgs F)
{
    const int t = blockIdx.x;
    const long long u0 = (long long)t * F.JS;
    const int g = owner_of(u0, F.U, F.G) + blockIdx.y;
    const long long ub = max(u0, (long long)g * F.U / F.G), ue = min(u0 + F.JS, (long long)(g + 1) * F.U / F.G);
    if (ub >= ue) return;
    const int b0 = (int)(ub - u0) * (F.JC / WAVE_B), b1 = min((int)(ue - u0) * (F.JC / WAVE_B), F.n_pad / WAVE_B);
    const int i = t * WAVE_TI + threadIdx.x;
    const long long ld = F.n_pad;
    float ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll 4
    for (int b = b0; b < b1; ++b) {
        const float* p = F.blk + 3ll * b * ld + i;
        ax += p[0];
        ay += p[ld];
        az += p[2 * ld];
    }
    part[(long long)blockIdx.y * ld + i] = make_float4(ax, ay, az, 0.f);
}

// The ordered kernel stays where the wave's units (one warp for 41 us when alone on its scheduler)
// are too few to fill the chip, and above 32,768 ions, where the block sums (12 n^2 / 128 bytes)
// outgrow L2 and the symmetric kernels with fixed-point sums are the default anyway.
// Whole steps, ordered and wave (with the fold): 6,000 ions 53 and 64 us, 7,000 61 and 66, 8,000
// 73 and 69, 9,000 93 and 88, 12,000 117 and 90, 16,000 181 and 139, 20,000 255 and 189, 32,000
// 612 and 396; the pair sums alone at 20,000 235 and 171, at 32,768 601 and 408.
bool wave_sums(const ForceArgs& F, int v)
{
    constexpr int MIN_PAD = 7680, MAX_PAD = 32768;
    return !F.sym && !F.cut && v >= 0 && v < num_force_variants() && force_variant(v).BT == WAVE_B &&
           F.TI == WAVE_TI && F.n_pad > MIN_PAD && F.n_pad <= MAX_PAD;
}

int launch_forces_wave(const Bufs& B, const ForceArgs& F, int v, cudaStream_t s)
{
    if (!wave_sums(F, v) || !F.sched) return (int)cudaErrorInvalidValue;
    int dev = 0, sms = 0, nb = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_forces_wave, WAVE_BT, 0);
    if (e != cudaSuccess) return (int)e;
    const int T = F.n_pad / WAVE_TI, warps = WAVE_BT / 32, units = T * (T + 1) / 2;
    k_forces_wave<<<std::min(std::max(nb, 1) * sms, (units + warps - 1) / warps), WAVE_BT, 0, s>>>(B.fpos, F);
    k_fold_blocks<<<dim3(T, F.W), WAVE_TI, 0, s>>>(B.part, F);
    return (int)cudaGetLastError();
}

}  // namespace od
