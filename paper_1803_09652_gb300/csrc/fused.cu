// Small batches: all phases of a force evaluation, or of a run of MD steps, in
// one launch.
//
// The passes of a small batch are shorter than what surrounds them: a step of
// 64 atoms takes 33 us as six launches, 1,024 atoms 37 us, of which each launch
// costs about 5 us whatever it does (its ramp, its cold constants and
// instructions, its last block's flush).  Here every replica has a
// thread-block cluster (8 warps a block, two blocks an SM) for the whole launch, and
// a phase ends with the cluster's barrier.  Clusters never wait for one
// another.  64 atoms: 20 us a step, 256: 26 (35 as six launches), one force
// evaluation of 237 atoms 31 us (40 as seven launches).  What is left is
// latency: of its 45,000 cycles the barriers with the reductions they wait for
// take 3,000 each, and a warp's one block 7,000 to 8,000, half of it its loads.
// Blocks of 8 warps rather than 16 spread a batch over all SMs (40 x 300 atoms:
// 36 against 42 us a step).
//
// Within a pass the warps of a group take its replica's tasks (64 x 32 blocks,
// the costly ones on the diagonal first, dealt out over the blocks) in rounds
// that the warps of a block run together, because the close pairs of a round's
// near blocks are evaluated by all of them: a diagonal block has ten times 32
// of them, 7,000 to 9,000 cycles for the warp that found them while the others
// had nothing left to do.  The blocks, their arithmetic and the
// fixed-point sums are those of the pass-by-pass launches: results are the same
// bit for bit.
#include "md_tiles.cuh"

namespace gbk {

constexpr int FUSED_SMEM = FUSED_WARPS * WARP_SMEM<Energy>;
static_assert(WARP_SMEM<Energy> >= WARP_SMEM<Chain> && WARP_SMEM<Energy> >= WARP_SMEM<Born>, "slot");

// Ends a phase of a replica: its cluster's barrier, which also orders its global
// memory accesses.
__device__ __forceinline__ void group_sync(int blocks) {
    if (blocks == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One task (row K against tile J); returns the close pairs left in the queue.
template <class P, int FLAGS>
__device__ __forceinline__ int round_task(const PairArgs& A, int r, int K, int J, int nb, int slot, int lane) {
    extern __shared__ __align__(16) unsigned char s_mem[];
    long long* sa = (long long*)(s_mem + slot) + (K & 1) * 64 * P::NQ;
#pragma unroll
    for (int q = 0; q < 2 * P::NQ; ++q) sa[32 * q + lane] = 0;
    __syncwarp();
    const int t0 = A.tile_off[r];
    float4 ih;
    const float4 il = row_box_lo(A, t0, K, nb, &ih);
    const BoxPair b = box_pair(il, ih, __ldcg(&A.boxes[2 * (t0 + J)]), __ldcg(&A.boxes[2 * (t0 + J) + 1]));
    const int tier = J < 2 * K + 2 ? 0 : row_tier<P, FLAGS>(A, b);
    if (tier > 0) {
        run_far<P, FLAGS, 1>(tier, A, r, 64 * K, J, 1u, slot);
        return 0;
    }
    return run_near<P, FLAGS, true>(A, r, K, J, 1u, P::RADIUS_CUT ? close_bound(b.amax, b.smax) : A.rep_sigma * A.rep_sigma,
                                    slot);
}

template <class P, int FLAGS>
__device__ __forceinline__ void round_pass(const FusedArgs& F, int r, int gw, int64_t base, int n, int nb, int warp,
                                           int lane) {
    typedef typename NearForm<P, FLAGS>::W W;
    constexpr bool CLOSE = NearForm<P, FLAGS>::CLOSE;
    __shared__ int2 s_close[FUSED_WARPS];          // close pairs left, K and J of the block they belong to
    const PairArgs& A = F.pa;
    const int slot = warp * WARP_SMEM<Energy>;
    const int t0 = F.task_off[r], nt = F.task_off[r + 1] - t0;
    for (int first = 0; first < nt; first += F.blocks * FUSED_WARPS) {
        const int at = first + gw;
        int K = 0, J = 0, cnt = 0;
        if (at < nt) {
            const int4 t = F.tasks[t0 + at];
            K = 2 * (t.y >> 2) + ((t.y & 3) == 2 ? 1 : 0);
            J = t.z;
            cnt = round_task<P, FLAGS>(A, r, K, J, nb, slot, lane);
        }
        if (CLOSE) {
            if (lane == 0) s_close[warp] = make_int2(cnt, (K << 16) | J);
            __syncthreads();
            const int2 c = s_close[lane & (FUSED_WARPS - 1)];
            int upto = (c.x + 31) >> 5;            // batches of the warps up to this lane's
#pragma unroll
            for (int o = 1; o < FUSED_WARPS; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, upto, o, FUSED_WARPS);
                if ((lane & (FUSED_WARPS - 1)) >= o) upto += v;
            }
            const int batches = __shfl_sync(0xffffffffu, upto, FUSED_WARPS - 1);
            for (int b = warp; b < batches; b += FUSED_WARPS) {
                const int w = __ffs(__ballot_sync(0xffffffffu, upto > b)) - 1;
                const int wc = __shfl_sync(0xffffffffu, c.x, w), kj = __shfl_sync(0xffffffffu, c.y, w);
                const int e = 32 * (b - (__shfl_sync(0xffffffffu, upto, w) - ((wc + 31) >> 5)));
                const Slot<W> S(w * WARP_SMEM<Energy>);
                run_close(A, S, (kj >> 16) & 1, e, wc, 64 * (kj >> 16), 32 * (kj & 0xffff), lane);
            }
            __syncthreads();
        } else {
            __syncwarp();
        }
        if (at < nt) {
            const Slot<W> S(slot);
            P::flush_i(A, base, n, 64 * K, lane, S.sa + (K & 1) * 64 * P::NQ);
            if (CLOSE && cnt && 32 * J + lane < n) W::flush_close(A, base + 32 * J + lane, S.jac, lane);
            __syncwarp();
        }
    }
}

template <int EFL>
__global__ void __launch_bounds__(32 * FUSED_WARPS, 2) k_fused(const __grid_constant__ FusedArgs P) {
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int r = blockIdx.x / P.blocks;
    // tasks and tiles are dealt out over the blocks first
    const int gw = blockIdx.x % P.blocks + P.blocks * warp, warps = P.blocks * FUSED_WARPS;
    const int64_t base = P.pa.atom_off[r];
    const int n = (int)(P.pa.atom_off[r + 1] - base), nb = (n + 31) >> 5;
    const u64 step0 = P.nsteps ? __ldcg(&P.md.ctr[0]) + (u64)P.step0 : 0;
    for (int s = 0;; ++s) {
        if (P.nsteps) {
            for (int u = gw; u < nb; u += warps) tile_halfsteps(P, r, u, lane, s > 0, s < P.nsteps, step0 + (u64)s + 1);
            if (s == P.nsteps) return;
        } else {
            for (int u = gw; u < nb; u += warps) tile_box_warp(P.pa, P.M, P.pa.tile_off[r] + u, lane);
        }
        group_sync(P.blocks);
        round_pass<Born, 0>(P, r, gw, base, n, nb, warp, lane);
        group_sync(P.blocks);
        for (int u = gw; u < nb; u += warps)
            if (32 * u + lane < n) born_finalize_atom(P.aa, base + 32 * u + lane, P.R_out);
        if (P.born_only) return;
        group_sync(P.blocks);
        round_pass<EnergyF<EFL>, EFL>(P, r, gw, base, n, nb, warp, lane);
        group_sync(P.blocks);
        for (int u = gw; u < nb; u += warps) atoms_chain_bonds(P, r, u, lane);
        group_sync(P.blocks);
        round_pass<Chain, 0>(P, r, gw, base, n, nb, warp, lane);
        group_sync(P.blocks);
        if (!P.nsteps) {
            for (int u = gw; u < nb; u += warps)
                if (32 * u + lane < n) forces_out_atom(P.aa, base + 32 * u + lane, P.F_fixed, P.F_out);
            return;
        }
    }
}

namespace {
typedef void (*FusedKernel)(FusedArgs);
FusedKernel fused_kernel(int flags) {
    switch (flags & (EF_REP | EF_SALT)) {
        case 0: return k_fused<0>;
        case EF_REP: return k_fused<EF_REP>;
        case EF_SALT: return k_fused<EF_SALT>;
        default: return k_fused<EF_REP | EF_SALT>;
    }
}
}  // namespace

cudaError_t fused_resident(int flags, int blocks, int* clusters) {
    const FusedKernel k = fused_kernel(flags);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(32 * FUSED_WARPS);
    cfg.dynamicSmemBytes = FUSED_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, k, &cfg);
}

cudaError_t launch_fused(const FusedArgs& a, int flags, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.M * a.blocks);
    cfg.blockDim = dim3(32 * FUSED_WARPS);
    cfg.dynamicSmemBytes = FUSED_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fused_kernel(flags), a);
}

}  // namespace gbk
