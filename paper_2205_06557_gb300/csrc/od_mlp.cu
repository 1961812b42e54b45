// The warm-start network's passes on the fifth-generation tensor cores.
//
// Every operation of the network but the weight gradients is local to a row tile of 16
// samples (128 rows: the pooled mean runs over the 8 rows of a sample), so one kernel takes
// a tile through all of them (k_mlp): the five layers with their activations and the set
// pooling, and for training the loss and the backward data products.  The activations
// stay in shared memory in the layout the next product reads; only what a caller or the weight
// gradients need goes to memory.
//
// What bounds it: a tile is 69 MFLOP of products against 528 KB of weights streamed from L2
// (forward; 125 MFLOP and 914 KB with the backward products) and ~1,000 accumulator columns read,
// activated, rounded and written back to shared memory by eight warps, which the products of the
// same tile cannot overlap (each layer needs the whole previous one).
//
// CTA of 320 threads, one per SM (128 KB of A operand, a three-stage ring of 32 KB weight chunks):
//   warp 9    one thread streams the weights: chunks of 64 K columns x N rows by TMA into the
//             ring, ahead of the products across layers and tiles
//   warp 8    one thread issues tcgen05.mma (M = 128, N = 256 or 16, K = 16) and commits
//   warps 0-7 epilogues: warp w reads accumulator lanes (rows) 32 (w % 4) .. + 31, columns
//             128 (w / 4) .. + 127 in blocks of 32, adds the bias, applies the relu (or the
//             saved relu mask), rounds to BF16 and writes the next product's A operand: K-major
//             128-byte swizzled chunks of 64 columns (row r at 128 r bytes, its 16-byte pieces
//             permuted by r mod 8)
// Sums that are rounded to BF16 afterwards (pooled means, their gradients) add in the order
// of the sample's rows, as the layer-by-layer kernels of od_sur.cu do.
//
// Measured against the layer-by-layer kernels on the same engine (calls through the C ABI with
// host arrays): forward of 16,384 samples 2,330 -> 260 us (kernels 510 -> 144 us; the rest was
// host repacking); loss and gradients of 128 samples 605 -> 160 us (39 launches -> 4, of which
// five serial column sums of 61 us), of 4,096 samples 10.7 -> 0.51 ms.
//
// Every wait is bounded: one that runs out sets bit 1 of *err and ends the CTA's work; loads in
// flight are waited for (again bounded) and the tensor memory is freed.
#include "od_mlp.cuh"

namespace od {
namespace mlp {

namespace {

using namespace tc;

constexpr int EPI_THREADS = 256, MMA_WARP = 8, TMA_WARP = 9, THREADS = 320;
constexpr int STAGES = 3;
constexpr int CHUNK = 64;                             // K columns per chunk
constexpr int REGION = TILE * CHUNK * 2;              // 16 KB: one chunk of the A operand
constexpr int A_BYTES = 8 * REGION;                   // up to K = 512
constexpr int STAGE_BYTES = H * CHUNK * 2;            // 32 KB
constexpr int SMEM_BYTES = A_BYTES + STAGES * STAGE_BYTES + 1024 + 128;
constexpr int STG_LD = 33;                            // staged 32 x 32 FP32 block (column reads)
static_assert(8 * 32 * STG_LD * 4 <= 4 * REGION, "staging fits the second half of the A operand");

// the products of a tile: weight map, first row of its box, K, N; forward 0-4, backward 5-9
// (8 is the second half of 7's 512 columns)
struct Step {
    int map, row0, K, N;
};
__device__ constexpr int NSTEP_F = 5, NSTEP_B = 10;
__device__ __forceinline__ Step step_of(int s)
{
    switch (s) {
    case 0: return {0, 0, K0, H};
    case 1: return {1, 0, H, H};
    case 2: return {2, 0, 2 * H, H};
    case 3: return {3, 0, H, H};
    case 4: return {4, 0, H, OUTP};
    case 5: return {5, 0, OUTP, H};
    case 6: return {6, 0, H, H};
    case 7: return {7, 0, H, H};
    case 8: return {7, H, H, H};
    default: return {8, 0, H, H};
    }
}

__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void commit_to(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* m, int c0, int c1, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void expect(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_store(const CUtensorMap* m, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"((uint64_t)m), "r"(c0),
                 "r"(c1), "r"(src)
                 : "memory");
}

// barrier of the epilogue warps; true in all of them if any passes true
__device__ __forceinline__ bool epi_any(bool v)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, 1, 256, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void st_shared16(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// byte address of the 16-byte piece holding columns col .. col + 7 (col a multiple of 8) of a row
__device__ __forceinline__ uint32_t a_piece(uint32_t sA, int row, int col)
{
    return sA + (uint32_t)((col >> 6) * REGION + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4));
}

// 32 columns of the thread's row, rounded to BF16, into the A operand
__device__ __forceinline__ void put_block(uint32_t sA, int row, int col, const float (&v)[32])
{
#pragma unroll
    for (int p = 0; p < 4; ++p)
        st_shared16(a_piece(sA, row, col + 8 * p), pack_bf16(v[8 * p], v[8 * p + 1]), pack_bf16(v[8 * p + 2], v[8 * p + 3]),
                    pack_bf16(v[8 * p + 4], v[8 * p + 5]), pack_bf16(v[8 * p + 6], v[8 * p + 7]));
}

// the warp's 32 x 32 FP32 block, row = lane, staged so that lane j can read column j
__device__ __forceinline__ void stage_block(float* stg, int lane, const float (&v)[32])
{
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 32; ++e) stg[lane * STG_LD + e] = v[e];
    __syncwarp();
}

// Four per-block values of a thread (relu mask words or partial sums of its half's four 32-column
// blocks) in registers: a loop over the blocks that is not unrolled takes the first and puts
// it back last, so that four turns leave them in place and nothing is indexed.
template <class T>
struct Ring4 {
    T a, b, c, d;
    __device__ __forceinline__ T turn(T last)
    {
        const T first = a;
        a = b, b = c, c = d, d = last;
        return first;
    }
};

// the accumulator columns [col, col + 32) of the warp's rows
__device__ __forceinline__ void read_acc(uint32_t taddr, float (&v)[32])
{
    uint32_t acc[32];
    tmem_issue<32>(taddr, acc);
    tmem_wait<32>(acc);
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
}

// bias and relu of a layer's columns (this warp's rows and half) into the A operand; the relu
// masks are kept for the backward pass
template <bool TRAIN>
__device__ __forceinline__ void relu_layer(uint32_t tq, uint32_t sA, int row, int half, const float* bias,
                                           Ring4<uint32_t>& mask)
{
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const int col = 128 * half + 32 * b;
        uint32_t acc[32];
        tmem_issue<32>(tq + (uint32_t)col, acc);
        float4 b4[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) b4[q] = __ldg((const float4*)(bias + col) + q);
        tmem_wait<32>(acc);
        float v[32];
        uint32_t bits = 0u;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const float4 bq = b4[e >> 2];
            const float be = (e & 3) == 0 ? bq.x : (e & 3) == 1 ? bq.y : (e & 3) == 2 ? bq.z : bq.w;
            v[e] = fmaxf(__uint_as_float(acc[e]) + be, 0.f);
            if (TRAIN) bits |= v[e] > 0.f ? 1u << e : 0u;
        }
        if (TRAIN) mask.turn(bits);
        put_block(sA, row, col, v);
    }
}

// the same for the second layer, whose outputs are also averaged over each sample's present rows
// (in row order) into columns 256 .. 511; m: the row's mask value, stg: the warp's staging in
// the second half of the operand
template <bool TRAIN>
__device__ __forceinline__ void relu_pool_layer(uint32_t tq, uint32_t sA, int row, int half, const float* bias,
                                                Ring4<uint32_t>& mask, float m, float* stg)
{
    const int lane = row & 31, row0 = row - lane;
    float n = 0.f;
    for (int k = 0; k < G; ++k) n += __shfl_sync(0xffffffffu, m, (lane & ~7) + k);
    Ring4<uint32_t> c01, c23;  // the lane's column's means (BF16) of the quarter's samples 0-1, 2-3
    c01.a = c01.b = c01.c = c01.d = c23.a = c23.b = c23.c = c23.d = 0u;
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const int col = 128 * half + 32 * b;
        float v[32];
        read_acc(tq + (uint32_t)col, v);
        uint32_t bits = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 bq = __ldg((const float4*)(bias + col) + q);
            v[4 * q] = fmaxf(v[4 * q] + bq.x, 0.f);
            v[4 * q + 1] = fmaxf(v[4 * q + 1] + bq.y, 0.f);
            v[4 * q + 2] = fmaxf(v[4 * q + 2] + bq.z, 0.f);
            v[4 * q + 3] = fmaxf(v[4 * q + 3] + bq.w, 0.f);
        }
        if (TRAIN) {
#pragma unroll
            for (int e = 0; e < 32; ++e) bits |= v[e] > 0.f ? 1u << e : 0u;
            mask.turn(bits);
        }
        put_block(sA, row, col, v);
        stage_block(stg, lane, v);
        float c[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            float sum = 0.f;
#pragma unroll
            for (int k = 0; k < G; ++k)
                sum = fmaf(__shfl_sync(0xffffffffu, m, 8 * s + k), stg[(8 * s + k) * STG_LD + lane], sum);
            const float ns = __shfl_sync(0xffffffffu, n, 8 * s);
            c[s] = ns > 0.f ? sum / ns : 0.f;
        }
        c01.turn(pack_bf16(c[0], c[1]));
        c23.turn(pack_bf16(c[2], c[3]));
    }
    epi_any(false);  // every warp's staging has been read
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const int col = H + 128 * half + 32 * b + lane;
        const uint32_t p01 = c01.turn(0u), p23 = c23.turn(0u);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const uint16_t c = (uint16_t)((s < 2 ? p01 : p23) >> (16 * (s & 1)));
#pragma unroll
            for (int k = 0; k < G; ++k)
                asm volatile("st.shared.b16 [%0], %1;" ::"r"(a_piece(sA, row0 + 8 * s + k, col & ~7) + 2u * (col & 7)),
                             "h"(c)
                             : "memory");
        }
    }
}

// one block of a layer's errors, masked by the layer's relu, into the A operand; the column
// sums (the lane's column over the warp's rows) go to the bias gradient
__device__ __forceinline__ void put_errors(uint32_t sA, int row, int col, float (&v)[32], Ring4<uint32_t>& mask,
                                           Ring4<float>& db, float* stg)
{
    const int lane = row & 31;
    const uint32_t bits = mask.turn(0u);
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = (bits >> e) & 1u ? v[e] : 0.f;
    put_block(sA, row, col, v);
    stage_block(stg, lane, v);
    float sum = 0.f;
#pragma unroll
    for (int r = 0; r < 32; ++r) sum += stg[r * STG_LD + lane];
    db.turn(db.a + sum);
}

__device__ __forceinline__ void error_layer(uint32_t tq, uint32_t sA, int row, int half, Ring4<uint32_t>& mask,
                                            Ring4<float>& db, float* stg)
{
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const int col = 128 * half + 32 * b;
        float v[32];
        read_acc(tq + (uint32_t)col, v);
        put_errors(sA, row, col, v, mask, db, stg);
    }
}

// the second layer's errors from dx3 = [dh2 | dc] (accumulator columns 0 .. 511): the pooled
// half's gradient, summed over the sample's present rows (in row order), is shared out to them
__device__ __forceinline__ void unpool_layer(uint32_t tq, uint32_t sA, int row, int half, Ring4<uint32_t>& mask,
                                             Ring4<float>& db, float m, float* stg)
{
    const int lane = row & 31;
    float n = 0.f;
    for (int k = 0; k < G; ++k) n += __shfl_sync(0xffffffffu, m, (lane & ~7) + k);
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const int col = 128 * half + 32 * b;
        float v[32];
        read_acc(tq + (uint32_t)(H + col), v);
        stage_block(stg, lane, v);
        float dc[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            dc[s] = 0.f;
#pragma unroll
            for (int k = 0; k < G; ++k)
                dc[s] = fmaf(__shfl_sync(0xffffffffu, m, 8 * s + k), stg[(8 * s + k) * STG_LD + lane], dc[s]);
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 4; ++s) stg[s * STG_LD + lane] = dc[s];
        __syncwarp();
        read_acc(tq + (uint32_t)col, v);
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] += n > 0.f ? m * stg[(lane >> 3) * STG_LD + e] / n : 0.f;
        put_errors(sA, row, col, v, mask, db, stg);
    }
}

template <bool TRAIN>
__global__ void __launch_bounds__(THREADS, 1) k_mlp(const __grid_constant__ FusedMaps M, FusedArgs A)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + A_BYTES + STAGES * STAGE_BYTES);  // a chunk has landed, per stage
    uint64_t* empty = full + STAGES;                                        // its products are done
    uint64_t* a_ready = empty + STAGES;                                     // the A operand is written
    uint64_t* acc_done = a_ready + 1;                                       // a layer's products are done
    uint32_t* tmem_slot = (uint32_t*)(acc_done + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NSTEP = TRAIN ? NSTEP_B : NSTEP_F;
    const uint32_t sA = smem_u32(smem), sB = sA + A_BYTES;

    if (threadIdx.x == 0) {
        for (int st = 0; st < STAGES; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        mbar_init(a_ready, EPI_THREADS);
        mbar_init(acc_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == TMA_WARP) {
        if (lane == 0) {
            int g = 0;  // chunks loaded
            bool ok = true;
            for (int t = blockIdx.x; t < A.tiles && ok; t += gridDim.x)
                for (int s = 0; s < NSTEP && ok; ++s) {
                    const Step S = step_of(s);
                    const int nch = (S.K + CHUNK - 1) / CHUNK;
                    for (int c = 0; c < nch && ok; ++c, ++g) {
                        const int st = g % STAGES, n = g / STAGES;
                        if (n > 0) ok = mbar_wait(&empty[st], (unsigned)(n - 1) & 1u);
                        if (!ok) break;
                        expect(&full[st], (uint32_t)(S.N * CHUNK * 2));
                        tma_load(sB + st * STAGE_BYTES, &M.w[S.map], c * CHUNK, S.row0, &full[st]);
                    }
                }
            if (!ok) atomicOr(A.err, 2);
            // no load is in flight when the CTA ends
            for (int k = g - STAGES < 0 ? 0 : g - STAGES; k < g; ++k)
                if (!mbar_wait(&full[k % STAGES], (unsigned)(k / STAGES) & 1u)) atomicOr(A.err, 2);
        }
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            int g = 0;
            unsigned ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < A.tiles && ok; t += gridDim.x)
                for (int s = 0; s < NSTEP && ok; ++s) {
                    const Step S = step_of(s);
                    if (s != 8) {
                        ok = mbar_wait(a_ready, ph);
                        ph ^= 1u;
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    const uint32_t idesc = instr_desc(TILE, S.N), d = tmem + (s == 8 ? (uint32_t)H : 0u);
                    for (int k0 = 0; k0 < S.K; k0 += CHUNK, ++g) {
                        const int st = g % STAGES;
                        ok = mbar_wait(&full[st], (unsigned)(g / STAGES) & 1u);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t a = sA + (k0 / CHUNK) * REGION, b = sB + st * STAGE_BYTES;
                        const int ks = min(CHUNK, S.K - k0) / 16;
                        for (int kk = 0; kk < ks; ++kk)
                            mma(d, smem_desc_sw128(a + 32u * kk), smem_desc_sw128(b + 32u * kk), idesc,
                                (k0 > 0 || kk > 0) ? 1u : 0u);
                        commit_to(&empty[st]);
                    }
                    if (ok && s != 7) commit_to(acc_done);
                }
            if (!ok) atomicOr(A.err, 2);
        }
    } else {
        const int quad = warp & 3, half = warp >> 2;
        const int row = 32 * quad + lane;
        const uint32_t tq = tmem + ((uint32_t)(32 * quad) << 16);
        float* stg = (float*)(smem + 4 * REGION) + warp * 32 * STG_LD;
        unsigned ph = 0;
        // relu masks of h1..h4 and bias gradients of dz1..dz4: this row (lane's column) of the
        // half's four 32-column blocks
        Ring4<uint32_t> rm[4];
        Ring4<float> db[4];
        float db5 = 0.f;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            rm[l].a = rm[l].b = rm[l].c = rm[l].d = 0u;
            db[l].a = db[l].b = db[l].c = db[l].d = 0.f;
        }

        // the accumulators are complete (and the A operand free to overwrite): true if not
        auto begin = [&]() {
            const bool ok = mbar_wait(acc_done, ph);
            ph ^= 1u;
            if (TRAIN && threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            if (!ok) atomicOr(A.err, 2);
            const bool bad = epi_any(!ok);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            return bad;
        };
        // hand the A operand to the products
        auto publish = [&]() {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            fence_async();
            mbar_arrive(a_ready);
        };
        // store nreg chunks of 64 columns of the A operand (training)
        auto store = [&](int map, int nreg, int r0) {
            fence_async();
            epi_any(false);
            if (threadIdx.x == 0) {
                for (int k = 0; k < nreg; ++k) tma_store(&M.act[map], sA + k * REGION, k * CHUNK, r0);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        };
        for (int t = blockIdx.x; t < A.tiles; t += gridDim.x) {
            const int r0 = t * TILE, gr = r0 + row;
            const bool live = gr < A.rows;
            const float m = live ? A.mask[gr] : 0.f;
            if (TRAIN) {  // the previous tile's last store has read the operand
                if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                epi_any(false);
            }
            if (half == 0) {
                float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                if (live)
#pragma unroll
                    for (int j = 0; j < IN; ++j) f[j] = A.x[(long long)gr * IN + j];
                const uint32_t p[4] = {pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]),
                                       pack_bf16(f[6], f[7])};
                st_shared16(a_piece(sA, row, 0), p[0], p[1], p[2], p[3]);
                st_shared16(a_piece(sA, row, 8), 0u, 0u, 0u, 0u);
                if (TRAIN) {
                    uint4* o = (uint4*)(A.x0 + (long long)gr * K0);
                    o[0] = make_uint4(p[0], p[1], p[2], p[3]);
                    o[1] = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            publish();
            if (begin()) break;
            relu_layer<TRAIN>(tq, sA, row, half, A.bias[0], rm[0]);
            publish();
            if (TRAIN) store(0, 4, r0);
            if (begin()) break;
            relu_pool_layer<TRAIN>(tq, sA, row, half, A.bias[1], rm[1], m, stg);
            publish();
            if (TRAIN) store(1, 8, r0);
            if (begin()) break;
            relu_layer<TRAIN>(tq, sA, row, half, A.bias[2], rm[2]);
            publish();
            if (TRAIN) store(2, 4, r0);
            if (begin()) break;
            relu_layer<TRAIN>(tq, sA, row, half, A.bias[3], rm[3]);
            publish();
            if (TRAIN) store(3, 4, r0);
            if (begin()) break;
            // output layer (and the loss)
            if (half == 0) {
                uint32_t acc[16];
                tmem_issue<16>(tq, acc);
                tmem_wait<16>(acc);
                const float4 b5 = __ldg((const float4*)A.bias[4]);
                const float y[4] = {__uint_as_float(acc[0]) + b5.x, __uint_as_float(acc[1]) + b5.y,
                                    __uint_as_float(acc[2]) + b5.z, __uint_as_float(acc[3]) + b5.w};
                if (live && A.y) ((float4*)A.y)[gr] = make_float4(y[0], y[1], y[2], y[3]);
                if (TRAIN) {
                    float d[4] = {0.f, 0.f, 0.f, 0.f}, l = 0.f;
                    if (m > 0.f) {
                        const float4 t4 = ((const float4*)A.tgt)[gr];
                        const float tt[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                        for (int o = 0; o < OUTR; ++o) {
                            const float e = y[o] - tt[o];
                            l += e * e;
                            d[o] = 2.f * e * A.inv_count;
                        }
                    }
                    A.row_loss[gr] = l * A.inv_count;
                    const uint32_t p0 = pack_bf16(d[0], d[1]), p1 = pack_bf16(d[2], d[3]);
                    st_shared16(a_piece(sA, row, 0), p0, p1, 0u, 0u);
                    st_shared16(a_piece(sA, row, 8), 0u, 0u, 0u, 0u);
                    uint4* o = (uint4*)(A.dy + (long long)gr * OUTP);
                    o[0] = make_uint4(p0, p1, 0u, 0u);
                    o[1] = make_uint4(0u, 0u, 0u, 0u);
                    // lanes 0-3 keep the column sums of d[0..3]
#pragma unroll
                    for (int o4 = 0; o4 < OUTR; ++o4) {
                        float sum = d[o4];
#pragma unroll
                        for (int o5 = 16; o5 > 0; o5 >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o5);
                        if (lane == o4) db5 += sum;
                    }
                }
            }
            if (!TRAIN) {
                // the accumulator has been read before the next tile's first product
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                continue;
            }
            publish();
            if (begin()) break;
            error_layer(tq, sA, row, half, rm[3], db[3], stg);  // dz4 = relu'(h4) dy W5
            publish();
            store(4, 4, r0);
            if (begin()) break;
            error_layer(tq, sA, row, half, rm[2], db[2], stg);  // dz3
            publish();
            store(5, 4, r0);
            if (begin()) break;
            unpool_layer(tq, sA, row, half, rm[1], db[1], m, stg);  // dz2
            publish();
            store(6, 4, r0);
            if (begin()) break;
            error_layer(tq, sA, row, half, rm[0], db[0], stg);  // dz1
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            store(7, 4, r0);
        }
        if (TRAIN) {
            if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            float* o = A.dbias + ((long long)blockIdx.x * QUADS + quad) * BIAS_LD;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                float* ol = o + l * H + 128 * half + lane;
                ol[0] = db[l].a, ol[32] = db[l].b, ol[64] = db[l].c, ol[96] = db[l].d;
            }
            if (half == 0 && lane < OUTP) o[4 * H + lane] = lane < OUTR ? db5 : 0.f;
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ------------------------------------------------------------ weight gradients
// dW[out][in] = sum over rows of dz[row][out] x[row][in]: the rows are the K dimension, so both
// operands are read as they lie in memory (MN-major: 64 rows x 64 columns boxes, 128-byte swizzle,
// 1,024 bytes between 8-row groups, 8,192 between 64-column blocks) and nothing is transposed.
// A CTA takes one 128 x (16 or 256) tile of one layer's dW (11 tiles over the five layers)
// and one of `splits` ranges of the rows, and writes an FP32 partial; k_grad_reduce adds
// them in order.  Four epilogue warps, one loading and one issuing thread, four stages of 48 KB.
constexpr int W_TILES = 11, W_THREADS = 192, W_STAGES = 4;
constexpr int BOX = 64 * 64 * 2;                         // 8 KB
constexpr int W_STAGE_BYTES = 6 * BOX;                   // 2 blocks of dz, up to 4 of x
constexpr int W_SMEM = W_STAGES * W_STAGE_BYTES + 1024 + 128;

struct WTile {
    int layer, m0, n0, N;
};
__device__ __forceinline__ WTile w_tile(int t)
{
    switch (t) {
    case 0: return {2, 0, 0, H};
    case 1: return {2, 128, 0, H};
    case 2: return {2, 0, H, H};
    case 3: return {2, 128, H, H};
    case 4: return {1, 0, 0, H};
    case 5: return {1, 128, 0, H};
    case 6: return {3, 0, 0, H};
    case 7: return {3, 128, 0, H};
    case 8: return {4, 0, 0, H};
    case 9: return {0, 0, 0, K0};
    default: return {0, 128, 0, K0};
    }
}

// shared-memory descriptor of an MN-major tile in the 128-byte swizzled layout
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)(BOX >> 4) << 16;      // leading byte offset: the next 64 columns
    d |= (uint64_t)(1024u >> 4) << 32;    // stride byte offset: the next 8 rows
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__global__ void __launch_bounds__(W_THREADS, 1)
    k_weight_grads(const __grid_constant__ GradMaps M, float* __restrict__ part, int rows, int splits, int* err)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + W_STAGES * W_STAGE_BYTES);
    uint64_t* empty = full + W_STAGES;
    uint64_t* acc_done = empty + W_STAGES;
    uint32_t* tmem_slot = (uint32_t*)(acc_done + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.x / W_TILES;
    const WTile T = w_tile(blockIdx.x % W_TILES);
    const int nch = (rows + 63) / 64;  // (rows past the last are zero errors in the padded buffers)
    const int c0 = (int)((long long)nch * split / splits), c1 = (int)((long long)nch * (split + 1) / splits);
    const int nb = (T.N + 63) / 64;
    const uint32_t ncols = T.N <= 32 ? 32u : 256u;
    const uint32_t s0 = smem_u32(smem);

    if (threadIdx.x == 0) {
        for (int st = 0; st < W_STAGES; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        mbar_init(acc_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 4) {
        if (lane == 0) {
            bool ok = true;
            int g = 0;
            for (int c = c0; c < c1 && ok; ++c, ++g) {
                const int st = g % W_STAGES, n = g / W_STAGES;
                if (n > 0) ok = mbar_wait(&empty[st], (unsigned)(n - 1) & 1u);
                if (!ok) break;
                const uint32_t a = s0 + st * W_STAGE_BYTES;
                expect(&full[st], (uint32_t)((2 + nb) * BOX));
                for (int k = 0; k < 2; ++k) tma_load(a + k * BOX, &M.dz[T.layer], T.m0 + 64 * k, c * 64, &full[st]);
                for (int k = 0; k < nb; ++k) tma_load(a + (2 + k) * BOX, &M.x[T.layer], T.n0 + 64 * k, c * 64, &full[st]);
            }
            if (!ok) atomicOr(err, 2);
            for (int k = g - W_STAGES < 0 ? 0 : g - W_STAGES; k < g; ++k)
                if (!mbar_wait(&full[k % W_STAGES], (unsigned)(k / W_STAGES) & 1u)) atomicOr(err, 2);
        }
    } else if (warp == 5) {
        if (lane == 0) {
            // both operands MN-major (bits 15 and 16)
            const uint32_t idesc = instr_desc(128, T.N) | (1u << 15) | (1u << 16);
            bool ok = true;
            for (int g = 0; g < c1 - c0; ++g) {
                const int st = g % W_STAGES;
                ok = mbar_wait(&full[st], (unsigned)(g / W_STAGES) & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = s0 + st * W_STAGE_BYTES, b = a + 2 * BOX;
                for (int kk = 0; kk < 4; ++kk)  // 16 rows: two 8-row groups
                    mma(tmem, smem_desc_mn(a + 2048u * kk), smem_desc_mn(b + 2048u * kk), idesc,
                        (g > 0 || kk > 0) ? 1u : 0u);
                commit_to(&empty[st]);
            }
            if (ok) commit_to(acc_done);
            else atomicOr(err, 2);
        }
    } else {
        const bool ok = mbar_wait(acc_done, 0u);
        if (!ok) atomicOr(err, 2);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int o = T.m0 + 32 * warp + lane;  // output row of dW
        const uint32_t tq = tmem + ((uint32_t)(32 * warp) << 16);
        float* dst = part + (long long)split * N_PARAMS + w_off(T.layer) + (long long)o * in_of(T.layer) + T.n0;
        const bool real = ok && o < out_of(T.layer);
        if (__any_sync(0xffffffffu, ok)) {
            if (T.N == K0) {
                uint32_t v[16];
                tmem_issue<16>(tq, v);
                tmem_wait<16>(v);
                if (real)
#pragma unroll
                    for (int q = 0; q < 4; ++q) ((uint4*)dst)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else {
                for (int b = 0; b < H / 32; ++b) {
                    uint32_t v[32];
                    tmem_issue<32>(tq + 32u * b, v);
                    tmem_wait<32>(v);
                    if (real)
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            ((uint4*)(dst + 32 * b))[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    }
}

// The gradient vector: weights from the split partials (four per thread, splits in order),
// biases from the fused pass's column sums (one warp per column, fixed tree).
constexpr int R_BT = 256;
constexpr int R_WBLOCKS = (N_PARAMS / 4 + R_BT - 1) / R_BT, R_BBLOCKS = (BIAS_LD + R_BT / 32 - 1) / (R_BT / 32);
static_assert(N_PARAMS % 4 == 0 && w_off(1) % 4 == 0 && w_off(2) % 4 == 0 && w_off(3) % 4 == 0 && w_off(4) % 4 == 0,
              "16-byte aligned layers");

__device__ __forceinline__ bool is_weight(int i)
{
#pragma unroll
    for (int l = 0; l < 5; ++l) {
        const int b = w_off(l) + out_of(l) * in_of(l);
        if (i >= b && i < b + out_of(l)) return false;
    }
    return true;
}

__global__ void __launch_bounds__(R_BT) k_grad_reduce(const float* __restrict__ part, int splits,
                                                      const float* __restrict__ dbias, int bias_rows,
                                                      float* __restrict__ grad)
{
    if (blockIdx.x < R_WBLOCKS) {
        const int i = 4 * (blockIdx.x * R_BT + threadIdx.x);
        if (i >= N_PARAMS || !is_weight(i)) return;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < splits; ++k) {
            const float4 p = __ldg((const float4*)(part + (long long)k * N_PARAMS + i));
            s.x += p.x, s.y += p.y, s.z += p.z, s.w += p.w;
        }
        *(float4*)(grad + i) = s;
        return;
    }
    const int c = (blockIdx.x - R_WBLOCKS) * (R_BT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= BIAS_LD) return;
    float s = 0.f;
    for (int r = lane; r < bias_rows; r += 32) s += dbias[(long long)r * BIAS_LD + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int l = c / H, j = c % H;  // the last 16 columns are layer 5's
    if (lane == 0) grad[w_off(l) + out_of(l) * in_of(l) + j] = s;
}

int ck(cudaError_t e) { return (int)e; }

}  // namespace

bool encode_maps(const __nv_bfloat16* const wb[5], const __nv_bfloat16* const wt[5], const Acts& A, int rows_pad,
                 FusedMaps& F, GradMaps& D)
{
    bool ok = true;
    for (int l = 0; l < 5; ++l) ok = ok && encode_tiled(&F.w[l], wb[l], out_of(l), in_of(l), out_of(l));
    ok = ok && encode_tiled(&F.w[5], wt[4], H, OUTP, H) && encode_tiled(&F.w[6], wt[3], H, H, H) &&
         encode_tiled(&F.w[7], wt[2], 2 * H, H, H) && encode_tiled(&F.w[8], wt[1], H, H, H);
    const __nv_bfloat16* const st[8] = {A.h1, A.x3, A.h3, A.h4, A.dz4, A.dz3, A.dz2, A.dz1};
    for (int k = 0; k < 8; ++k) ok = ok && encode_tiled(&F.act[k], st[k], rows_pad, k == 1 ? 2 * H : H, TILE);
    const __nv_bfloat16* const dz[5] = {A.dz1, A.dz2, A.dz3, A.dz4, A.dy};
    const __nv_bfloat16* const x[5] = {A.x0, A.h1, A.x3, A.h3, A.h4};
    for (int l = 0; l < 5; ++l)
        ok = ok && encode_tiled(&D.dz[l], dz[l], rows_pad, out_of(l), 64) && encode_tiled(&D.x[l], x[l], rows_pad, in_of(l), 64);
    return ok;
}

int launch_forward(const FusedMaps& M, const FusedArgs& A, int sms, cudaStream_t s)
{
    const cudaError_t e = cudaFuncSetAttribute(k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return ck(e);
    k_mlp<false><<<A.tiles < sms ? A.tiles : sms, THREADS, SMEM_BYTES, s>>>(M, A);
    return ck(cudaGetLastError());
}

int launch_forward_backward(const FusedMaps& M, const FusedArgs& A, int sms, int* ctas, cudaStream_t s)
{
    const cudaError_t e = cudaFuncSetAttribute(k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return ck(e);
    *ctas = A.tiles < sms ? A.tiles : sms;
    k_mlp<true><<<*ctas, THREADS, SMEM_BYTES, s>>>(M, A);
    return ck(cudaGetLastError());
}

// Row ranges: enough CTAs for the chip.  The tensor memory accumulator rounds towards zero, which
// takes ~1e-9 of a sum per row off a chain, so gradients summed over ranges move away from those
// of a single chain as the rows grow (they get more exact).  They stay within 1.5e-5 of it: sms / 11
// ranges up to 12,800 rows (1,600 samples: 1.4e-5; 2,048: 1.7e-5), two up to 20,480 (2,400
// samples: 1.35e-5; 4,096: 2.1e-5), one beyond (4,096 samples, loss and gradients: 511 us
// against 410 with two ranges).
int grad_splits(int rows, int sms)
{
    const int nch = (rows + 63) / 64, want = rows > 20480 ? 1 : rows > 12800 ? 2 : sms / W_TILES;
    return nch < want ? nch : want < 1 ? 1 : want;
}

// The ranges fall as the rows grow, so a small batch may need more of them than a full one.
int max_grad_splits(int max_rows, int sms)
{
    const int nch = (max_rows + 63) / 64, most = sms / W_TILES > 2 ? sms / W_TILES : 2;
    return nch < most ? nch : most;
}

int launch_weight_grads(const GradMaps& M, float* part, int rows, int splits, int* err, cudaStream_t s)
{
    const cudaError_t e = cudaFuncSetAttribute(k_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, W_SMEM);
    if (e != cudaSuccess) return ck(e);
    k_weight_grads<<<W_TILES * splits, W_THREADS, W_SMEM, s>>>(M, part, rows, splits, err);
    return ck(cudaGetLastError());
}

int launch_grad_reduce(const float* part, int splits, const float* dbias, int bias_rows, float* grad, cudaStream_t s)
{
    k_grad_reduce<<<R_WBLOCKS + R_BBLOCKS, R_BT, 0, s>>>(part, splits, dbias, bias_rows, grad);
    return ck(cudaGetLastError());
}

}  // namespace mlp
}  // namespace od
