// MD work on one 32-atom tile by one warp, shared by the kernels that run
// several phases of a step in one launch (persist.cu, fused.cu).
#pragma once

#include "atoms_impl.cuh"
#include "pairs_impl.cuh"

namespace gbk {

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Phase 0 on tile u of replica r.  second: close the previous step (force
// from the accumulators, kick).  first: open step `step` (B A O A with the
// same force) and rebuild the tile's box; otherwise store the force.
template <class Args>
__device__ __forceinline__ void tile_halfsteps(const Args& P, int r, int u, int lane, bool second,
                                               bool first, u64 step) {
    const MDArgs& m = P.md;
    const int64_t N = P.pa.N;
    const int64_t base = P.pa.atom_off[r];
    const int n = (int)(P.pa.atom_off[r + 1] - base);
    const int i = 32 * u + lane;
    if (i < n) {
        const int64_t g = base + i;
        float4 v = __ldcg(&m.vel[g]);
        float4 f;
        if (second) {
            f = make_float4((float)unfix(__ldcg(&P.aa.F_acc[g])), (float)unfix(__ldcg(&P.aa.F_acc[N + g])),
                            (float)unfix(__ldcg(&P.aa.F_acc[2 * N + g])), 0.0f);
            P.aa.F_acc[g] = 0;
            P.aa.F_acc[N + g] = 0;
            P.aa.F_acc[2 * N + g] = 0;
            v.x = fmaf(m.h * m.inv_m, f.x, v.x);
            v.y = fmaf(m.h * m.inv_m, f.y, v.y);
            v.z = fmaf(m.h * m.inv_m, f.z, v.z);
        } else {
            f = __ldcg(&m.force[g]);
        }
        if (first) {
            float4 x = __ldcg(&m.xyzq[g]);
            baoab_first(m, x, v, f, md_normals(m.seed, m.rep_base + (u64)r, step, (u64)i));
            m.xyzq[g] = x;
        } else {
            m.force[g] = f;
        }
        m.vel[g] = v;
    }
    if (first) tile_box_warp(P.pa, P.M, P.pa.tile_off[r] + u, lane);
}

// Phase 4 on atoms 32u .. 32u+31 of replica r: chain factor, chain bonds.
template <class Args>
__device__ __forceinline__ void atoms_chain_bonds(const Args& P, int r, int u, int lane) {
    const int64_t base = P.pa.atom_off[r];
    const int n = (int)(P.pa.atom_off[r + 1] - base);
    const int i = 32 * u + lane;
    if (i >= n) return;
    double R;
    chain_bond_atom(P.aa, P.md.xyzq, P.md.bond_k, P.md.bond_r0, base, i, n, &R);
}

}  // namespace gbk
