// Persistent MD kernel: several BAOAB steps of the whole batch in one launch,
// scheduled as a stream of warp-sized work items with per-replica
// dependencies instead of global barriers.
//
// Each MD step s of replica r runs six phases:
//   0  close step s-1 (total force -> kick), open step s (B A O A), rebuild
//      the tile's bounding box                              [item: 32-atom tile]
//   1  Born integrals                                       [item: pair task]
//   2  Born radii                                           [item: 32 atoms]
//   3  GB + Coulomb forces, dE/dR, soft repulsion           [item: pair task]
//   4  chain factors, chain bonds                           [item: 32 atoms]
//   5  Born chain-rule forces                               [item: pair task]
// and the launch ends with phase 0 of step nsteps (kick only; the forces are
// stored for the next launch).  Items are numbered step-major, then
// phase-major, then replica-major, and warps take them in that order from a
// global counter.  Phase p > 0 of (s, r) waits until all phase p-1 items of
// (s, r) are done, phase 0 of (s, r) until all phase 5 items of (s-1, r) are
// done.  Every wait is on items that come earlier in the order, which some
// running warp has already taken and will finish, so the schedule cannot
// deadlock and needs no co-residency.  While the last replica of a pass is
// still finishing, other warps already work on the next pass of the first
// replicas: the pass tails of a small batch overlap.
//
// Waits are bounded: after P.spin_limit polls (2^22 by default, about a
// quarter of a second; gb_set_wait_limit) the warp records GB_ERR_TIMEOUT and
// stops taking work; the others then see the error word, or time out on it,
// and stop too, so the launch always ends and the context stays usable.
#include "md_tiles.cuh"

namespace gbk {

constexpr int PERSIST_THREADS = 128;
constexpr int PERSIST_SMEM = WARP_SMEM<Energy>;   // the largest of the three passes' slots
static_assert(PERSIST_SMEM >= WARP_SMEM<Chain> && PERSIST_SMEM >= WARP_SMEM<Born>, "slot");

// Lane 0 waits until *ctr >= target; returns false when the wait gave up or
// another warp reported an error.
__device__ __forceinline__ bool wait_count(const unsigned* ctr, unsigned target, int* err, unsigned limit,
                                           int lane) {
    int ok = 1;
    if (lane == 0) {
        unsigned it = 0;
        while (ld_acquire(ctr) < target) {
            if (*(volatile int*)err != 0) { ok = 0; break; }
            if (++it > limit) {
                atomicCAS(err, 0, GB_ERR_TIMEOUT);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();
    return ok != 0;
}

// Four blocks an SM at 128 registers: at 80 (six blocks, of which shared memory
// holds five) the pair code spilled 700 to 980 bytes a thread.  us an MD step with
// 80 / 96 / 128 registers: 8 x 2048 176 / 164 / 153, 16 x 4096 801 / 746 / 698, 4 x 300
// 70 / 64 / 55, 8 x 25000 8160 / 7830 / 7780.  SMALL as in walk_task: 158 and 720 us
// for the first two without it.
template <int REP, bool SMALL>
__global__ void __launch_bounds__(PERSIST_THREADS, 4) k_md_persist(const __grid_constant__ PersistArgs P) {
    constexpr int EFL = REP ? EF_REP : 0;
    const int lane = threadIdx.x & 31;
    const int slot = (threadIdx.x >> 5) * PERSIST_SMEM;
    const unsigned per_step = (unsigned)P.phase_base[6];
    const unsigned total = per_step * (unsigned)P.nsteps + (unsigned)P.phase_base[1];
    const u64 step0 = __ldcg(&P.md.ctr[0]) + (u64)P.step0;
    for (;;) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(P.head, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= total) break;
        const int s = (int)(item / per_step);
        const unsigned rem = item - (unsigned)s * per_step;
        int p = 0;
        while (p < 5 && rem >= (unsigned)P.phase_base[p + 1]) ++p;
        const int* off = P.phase_off + p * (P.M + 1);
        const int x = (int)(rem - (unsigned)P.phase_base[p]);
        int lo = 0, hi = P.M;                  // replica with off[lo] <= x < off[lo + 1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= x) lo = mid;
            else hi = mid;
        }
        const int r = lo, u = x - off[r];
        // dependency: the previous phase of (s, r) -- or phase 5 of (s-1, r)
        bool ok = true;
        if (p > 0) {
            ok = wait_count(&P.done[(p - 1) * P.M + r], (unsigned)(s + 1) * (unsigned)P.count[(p - 1) * P.M + r],
                            P.err, P.spin_limit, lane);
        } else if (s > 0) {
            ok = wait_count(&P.done[5 * P.M + r], (unsigned)s * (unsigned)P.count[5 * P.M + r], P.err,
                            P.spin_limit, lane);
        }
        if (!ok) break;
        switch (p) {
            case 0: tile_halfsteps(P, r, u, lane, s > 0, s < P.nsteps, step0 + (u64)s + 1); break;
            case 1: walk_task<Born, 0, SMALL>(P.pa, P.tasks[P.task_off[r] + u], slot, lane); break;
            case 2: {
                const int64_t base = P.pa.atom_off[r];
                const int i = 32 * u + lane;
                if (i < (int)(P.pa.atom_off[r + 1] - base)) born_finalize_atom(P.aa, base + i, P.R_out);
                break;
            }
            case 3: walk_task<EnergyF<EFL>, EFL, SMALL>(P.pa, P.tasks[P.task_off[r] + u], slot, lane); break;
            case 4: atoms_chain_bonds(P, r, u, lane); break;
            default: walk_task<Chain, 0, SMALL>(P.pa, P.tasks[P.task_off[r] + u], slot, lane); break;
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(&P.done[p * P.M + r], 1u);
    }
}

namespace {
constexpr size_t PERSIST_BLOCK_SMEM = (PERSIST_THREADS / 32) * PERSIST_SMEM;
typedef void (*PersistKernel)(PersistArgs);
PersistKernel persist_kernel(int rep, bool small) {
    if (small) return rep ? k_md_persist<1, true> : k_md_persist<0, true>;
    return rep ? k_md_persist<1, false> : k_md_persist<0, false>;
}
}  // namespace

cudaError_t persist_occupancy(int rep, bool small, int* blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, persist_kernel(rep, small), PERSIST_THREADS,
                                                         PERSIST_BLOCK_SMEM);
}

cudaError_t launch_persist(const PersistArgs& a, int rep, bool small, int grid, cudaStream_t s) {
    // queue head and the per-(phase, replica) completion counters start at zero
    cudaError_t e = cudaMemsetAsync(a.head, 0, sizeof(unsigned) * (1 + 6 * (size_t)a.M), s);
    if (e != cudaSuccess) return e;
    persist_kernel(rep, small)<<<grid, PERSIST_THREADS, PERSIST_BLOCK_SMEM, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gbk
