// bz_lzbatch.cuh -- the active-node kernel over the cells of many instances.
#pragma once

#include "bz_ahead.cuh"

namespace bzk {

// ---------------------------------------------------------------------
// Persistent active-node schedule: every instance keeps its own active-node
// step (bz_lazy.cuh: sample plan, compact arrays, deferred correction), and
// one launch per kernel class runs that step for all instances.  The per-step
// plan kernels are flattened over the samples (or take one CTA per
// instance); the per-cell kernel k_lz runs as persistent CTAs that claim
// segments (an instance and a range of its cell groups) from a counter, one
// pipeline per segment.  An instance whose step has more active nodes than
// its compact arrays hold takes the 4-node-vector kernel instead (a gated
// chain that does nothing otherwise).
// ---------------------------------------------------------------------
struct LzInst {
    Geo g;                       // the instance's problem (the 4-node kernel's plan order)
    LzArgs a[2];                 // arguments of k_lz for a state of step parity 0 and 1
    int64_t *step;               // device step counter
    float *h[2], *mu[2];         // state buffers and their pending corrections, by step parity
    float *ghost;
    double *nw;
    int4 *idx;                   // the step's sample set (node indices, logical order)
    PlanA<float, int> *pa;
    ushort4 *qc;                 // compact indices of the samples' nodes
    int *flag, *cidx, *count, *cursor, *rowend;
    // the 4-node-vector fallback
    Map4 map;
    ushort4 *pidx16;
    PlanA<float, uint16_t> *pa16;
    int *sc_count, *sc_cursor, *sc_meta;
    uint32_t *sc_ent;
    AheadPlans ahead;            // the instance's plans built ahead (K = 0: none)
};

// The per-cell step of every instance: persistent CTAs claim segments
// (x: instance, y: first group, z: groups, w: stride between them) from *next
// until none are left.  The segments of an instance are claimed one after
// the other, so they run at the same time and interleave over its groups
// (neighbouring cells are streamed together and their slabs shared in L2).
// Groups of four cells; one launch per velocity grid (NV: its axis length),
// sized for that grid.
template <int NV>
__global__ void __launch_bounds__(lz_threads(lz_stream_threads(NV)), 1) kbl_lz(const LzInst *__restrict__ inst,
                                                       const int4 *__restrict__ segs, int nseg,
                                                       int *__restrict__ next)
{
    extern __shared__ __align__(16) char smem_raw[];
    __shared__ int s_seg;
    __shared__ Geo s_g;                     // the segment's problem and arguments
    __shared__ LzArgs s_a;
    for (;;) {
        __syncthreads();                    // the last segment's shared memory is free
        if (threadIdx.x == 0) s_seg = atomicAdd(next, 1);
        __syncthreads();
        const int sg = s_seg;
        if (sg >= nseg) break;
        const int4 q = segs[sg];
        const LzInst &b = inst[q.x];
        if (threadIdx.x == 0) {
            s_g = b.g;
            s_a = b.a[*b.step & 1];
        }
        __syncthreads();
        lz_run<4, NV, false, lz_stream_threads(NV)>(s_g, s_a, smem_raw, q.y, q.w, q.z);
    }
}

}  // namespace bzk
