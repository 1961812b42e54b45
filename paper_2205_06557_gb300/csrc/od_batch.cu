// Batched persistent step: many independent runs of uneven ion count advance one
// step in ONE kernel launch (replayed from a CUDA graph).
//
// Every run's step is split into tasks (BatchTask): scan tiles of 128 ions; pair units of one
// target tile x one source chunk (or tile pairs); side tiles of 128 ions (the ion terms and
// the grain sums, which need the positions but not the pair forces); a grain tail; kick tiles.
// A persistent grid of at most the resident number of CTAs takes tasks from a global
// counter: the runs' pair units one run after the other, each run's scan tiles well ahead of them
// and its side tiles between them, then all tails and kick tiles.  A task first waits until the
// counters of the kinds it depends on (of its run) reach their targets: pair units and side
// tiles for the scan, the tail for the side tiles, the kick for the pair units and the side
// tiles; every task waited for was handed out earlier to a CTA that is running, so the waits
// end (and each is bounded anyway: it gives up after spin_limit polls and sets an error).
// The counters only grow (target = (batch step + 1) x tasks of the kind), so nothing
// is reset between launches; the last CTA to leave advances the batch step.  A new plan
// (other numbers of tasks and CTAs) starts them again.
// What bounds it: the latency of a step's chain (scan, pair units, kick) and, between, the FP32 pipe
// for the pair units and the FP64 pipe for the rest, which is why the two are mixed.  48 runs of
// 2,171 ions (tile pairs of 256 ions), per step: 223 us with the ion terms and grain sums
// inside the kick tiles, 198 with side tiles of their own after all pair units, 181 with the
// side tiles between the pair units and polls at most 256 ns apart.  32 runs of 6,283: 578 -> 553.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "od_device.cuh"

namespace od {

constexpr int BATCH_BT = BATCH_TILE;

__device__ __forceinline__ unsigned long long ld_acquire_u64c(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// The ion terms and the grain side of one tile (kick_body<..., true> and dust_body follow): what
// k_ion_terms and k_grains do for a single run.
template <int BT>
__device__ __forceinline__ void side_tile(const Phys& P, const Bufs& B, int tile)
{
    Ctrl* C = B.ctrl;
    const int i = tile * BT + threadIdx.x;
    const bool live = i < C->n_cur;
    const long long step = B.felt->step, cap = B.cap;
    const int buf = (int)((step + 1) & 1);
    const uint32_t sn = (uint32_t)(step + 1);
    double x = 0, y = 0, z = 0;
    int coll = 0;
    if (live) {
        const double* X = B.x[buf];
        x = X[i], y = X[cap + i], z = X[2 * cap + i];
        const unsigned long long id = B.id[buf][i];
        double* T = B.pre;
        double a, b, c;
        if (P.cp_on) {
            close_pairs_of<1>(P, B, buf, i, x, y, z, a, b, c);
            T[i] = a, T[cap + i] = b, T[2 * cap + i] = c;
        }
        ion_field(P, x, y, z, a, b, c);
        T[3 * cap + i] = a, T[4 * cap + i] = b, T[5 * cap + i] = c;
        const uint4 w = philox(P, id, sn, ST_COLL);
        if ((unsigned long long)w.x < P.Tcoll) {
            collision_velocity(P, id, sn, a, b, c);
            B.coll_v[i] = a, B.coll_v[cap + i] = b, B.coll_v[2 * cap + i] = c;
            coll = 1;
        }
    }
    const unsigned bc = __ballot_sync(0xffffffffu, coll);
    if ((threadIdx.x & 31) == 0 && bc) atomicAdd(&C->ev_step[12], __popc(bc));
    grain_sums<BT>(P, B, live, x, y, z, tile);
}

// bounded wait of the whole CTA for a run's counter to reach target
__device__ __forceinline__ void wait_count(const unsigned long long* cnt, unsigned long long target, long long spin_limit,
                                           BatchCtrl* bc)
{
    if (threadIdx.x == 0) {
        long long spins = 0;
        unsigned ns = 64;
        while (ld_acquire_u64c(cnt) < target) {
            if (++spins > spin_limit) {
                atomicOr(&bc->err, ERR_TIMEOUT);
                break;
            }
            __nanosleep(ns);
            if (ns < 256) ns *= 2;
        }
    }
    __syncthreads();
}

// A task is (kind << 28 | run, index within the kind).  Tuning launches hold only pair units
// and BT_FORCES kick tiles (accelerations only: no velocity update, no collisions) on counters
// of their own; their pair units do not wait, so the runs' states are not changed.
// Held to 128 registers (four CTAs per SM), the units of eight targets per lane to 168
// (three; forces of 12 runs of 1e4 to 2e5 ions: 30.07 -> 29.11 ms).
template <int IPT>
__global__ void __launch_bounds__(BATCH_BT, 65536 / (BATCH_BT * (IPT == 8 ? 168 : 128)))
    k_batch_step(const RunDesc* __restrict__ runs, const int2* __restrict__ tasks, long long T, BatchCtrl* bc,
                 unsigned long long* done, int R, long long spin_limit, int tune)
{
    __shared__ SymShared<BATCH_BT / 32, BATCH_BT * IPT> sym;
    __shared__ long long s_task;
    const unsigned long long bstep = bc->step;
    // every launch draws exactly T + gridDim.x tickets (T tasks plus one failing draw per CTA)
    const unsigned long long base = bstep * (unsigned long long)(T + gridDim.x);
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_task = (long long)(atomicAdd(&bc->task_next, 1ull) - base);
        __syncthreads();
        const long long t = s_task;
        if (t >= T) break;
        const int2 tk = tasks[t];
        const int kind = (unsigned)tk.x >> 28, r = tk.x & ((1 << 28) - 1);
        const RunDesc& d = runs[r];
        unsigned long long* cnt = done + r;  // [0] scan tiles, [R] pair units, [2 R] side tiles
        const unsigned long long turn = bstep + 1;
        switch (kind) {
        case BT_SCAN: push_scan_body<BATCH_BT>(d.P, d.B, d.nA, 1.4426950408889634 * d.P.lam_inv, tk.y); break;
        case BT_PAIR:
            if (!tune) wait_count(cnt, turn * d.nA, spin_limit, bc);
            if (d.F.sym) {
                int I, J;
                tri_unit(tk.y, d.F.JS, I, J);
                sym2_unit<BATCH_BT, IPT>(d.B.fpos, d.F, I, J, sym);
            } else {
                forces_unit<BATCH_BT, IPT>(d.B.fpos, d.B.part, d.F, tk.y / d.F.JS, tk.y % d.F.JS, sym.sj);
            }
            break;
        case BT_SIDE:
            wait_count(cnt, turn * d.nA, spin_limit, bc);
            side_tile<BATCH_BT>(d.P, d.B, tk.y);
            break;
        case BT_TAIL:
            wait_count(cnt + 2 * R, turn * d.nK, spin_limit, bc);
            dust_body<false>(d.P, d.B, d.nK, 0);
            break;
        case BT_KICK:
            wait_count(cnt + R, turn * (unsigned long long)d.F.U, spin_limit, bc);
            wait_count(cnt + 2 * R, turn * d.nK, spin_limit, bc);
            kick_body<BATCH_BT, 1, true>(d.P, d.B, d.F, tk.y);
            break;
        default:
            wait_count(cnt + R, turn * (unsigned long long)d.F.U, spin_limit, bc);
            kick_body<BATCH_BT, 1>(d.P, d.B, d.F, tk.y);
            break;
        }
        if (kind > BT_SIDE) continue;  // nothing in this launch waits for it
        // publish completion of this task to the run's counter of its kind
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(cnt + (long long)kind * R, 1ull);
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&bc->exit_count, 1u) == gridDim.x - 1) {
            bc->exit_count = 0u;
            bc->step = bstep + 1;
        }
    }
}

static void* batch_fn(int ipt)
{
    switch (ipt) {
    case 2: return (void*)k_batch_step<2>;
    case 4: return (void*)k_batch_step<4>;
    default: return (void*)k_batch_step<8>;
    }
}

int batch_blocks_per_sm(int ipt)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_fn(ipt), BATCH_BT, 0) != cudaSuccess) return 1;
    return nb > 0 ? nb : 1;
}

int launch_batch(int ipt, int grid, const RunDesc* runs, const int2* tasks, long long T, BatchCtrl* bc,
                 unsigned long long* done, int R, long long spin_limit, int tune, cudaStream_t s)
{
    switch (ipt) {
    case 2:
        k_batch_step<2><<<grid, BATCH_BT, 0, s>>>(runs, tasks, T, bc, done, R, spin_limit, tune);
        break;
    case 4:
        k_batch_step<4><<<grid, BATCH_BT, 0, s>>>(runs, tasks, T, bc, done, R, spin_limit, tune);
        break;
    default:
        k_batch_step<8><<<grid, BATCH_BT, 0, s>>>(runs, tasks, T, bc, done, R, spin_limit, tune);
        break;
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : (int)e;
}

// the pair partition of one run inside a batch: tiles of BATCH_BT * ipt targets, source
// chunks of jc, every unit its own task (G = U, slot = chunk); jc = 0 selects the
// symmetric tile pairs of the packed kernel
ForceArgs batch_plan(int N, int ipt, int jc)
{
    ForceArgs F{};
    F.TI = BATCH_BT * ipt;
    F.n_pad = N == 0 ? 0 : (N + F.TI - 1) / F.TI * F.TI;
    if (F.n_pad == 0) return F;
    if (jc == 0) {
        // symmetric tile pairs (I, J >= I) into the fixed-point accumulators
        const int T = F.n_pad / F.TI;
        F.sym = 1;
        F.JC = F.TI;
        F.JS = T;
        F.W = 0;
        F.U = (long long)T * (T + 1) / 2;
        F.G = (int)F.U;
        return F;
    }
    F.JC = std::max(BATCH_BT, std::min(jc, F.n_pad) / BATCH_BT * BATCH_BT);
    F.JS = (F.n_pad + F.JC - 1) / F.JC;
    F.U = (long long)(F.n_pad / F.TI) * F.JS;
    F.G = (int)F.U;
    F.W = F.JS;
    return F;
}

}  // namespace od
