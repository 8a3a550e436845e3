// bz_lazy.cuh -- FP32 step on the active velocity nodes, correction deferred.
//
// Same mathematics as k_cell4 (Eqs. streaming2D, monteCarloInt,
// collision_step, rinorm_a, correzione, densita..sforzi), organised around two
// facts:
//
// * The Monte Carlo terms of a step touch only the nodes that one of its
//   shared samples maps to (v, v1, v*, v1*): for Maxwellian draws a small
//   fraction of the grid (about 7% of 32^3 at 2x10^4 samples).  Every other
//   node keeps h_c = h~.  The per-step plan lists those "active" nodes once
//   (compact index m), and the collision terms of every cell work on arrays
//   of M entries instead of the whole velocity slab.
// * The correction h^{n+1} = h_c + (1 + eps h_c)(mu . psi) needs mu, which
//   needs the moments of every node.  Instead of holding the whole slab until
//   mu is known, the step stores h_c and the cell's mu; whoever reads the
//   state next (the next step's streaming, the walls, a state copy) applies
//   the correction on the fly.  The state is therefore the pair (h_c, mu);
//   mu = 0 is an ordinary state.
//
// Without the slab a CTA needs two compact arrays, so two CTAs share an SM
// and each works on G cells at once: the G values of a node are adjacent, so
// one vector access serves all G cells and every collision term is decoded
// once per G cells.
//
// The collision terms are applied as a pull: the plan sorts the terms
// (destination, sample, sign) by destination and gives each thread a run of
// them; a term carries the byte offsets of the sample's two pre-collision
// nodes and its signed weight, so the thread recomputes the sample's product
// from h~ and sums a destination's terms in registers.  Floating-point
// arithmetic on node pairs uses the packed FP32x2 instructions.
//
// The conserved-moment sums of N_c and the output moments come from 26
// monomial sums (degree <= 4) of N = w h~ over all nodes, taken while
// streaming, plus the same sums of the collision increment over the active
// nodes.  If a step has more active nodes than the kernel's arrays hold
// (mcap), the kernel returns at once and the k_cell4 path computes the step.
#pragma once

#include "bz_cell4.cuh"

#include <type_traits>

namespace bzk {

constexpr int kLzMono = 26;        // monomial sums per cell
constexpr int kLzX = 30;           // with v^2, v_x v^2, v_y v^2, v_z v^2
// Threads of the collision role, and of the streaming role (ST, a template
// argument of the kernel).  256 streaming threads leave 128 registers a
// thread; with 512 (80 registers) a stage covers up to twice the jx-planes or
// more, so that the streaming of a cell takes fewer stages, but each stage of
// the ring is larger.  512 pay only where they keep a larger share of the
// threads busy: at 24 nodes per axis a stage has 432 quads (3 planes) against
// 144 (1 plane of 256 threads).  k_lz with 256 / 512 streaming threads: 128^2 x
// 24^3 989 / 821 us; 128^2 x 20^3 580 / 598, 128^2 x 16^3 407 / 480, 96^2 x 28^3 757 /
// 780, 128^2 x 12^3 284 / 346 us.
constexpr int kLzCollT = 256;
constexpr int kLzMaxStreamT = 512;
__host__ __device__ constexpr int lz_threads(int ST) { return ST + kLzCollT; }
constexpr int kLzDParts = 8;       // slots of the increment sums per cell
constexpr int kLzMaxG = 4;         // cells per CTA group
constexpr int kLzMaxN = 32;        // velocity nodes per axis (N^2 / 4 <= 256)
constexpr int kLzMaxStages = 5;    // streaming stages staged per thread (at least kLzMinStages)
constexpr int kLzMinStages = 3;    // (two: 256^2 x 32^3 6.28 -> 6.76 ms)
constexpr unsigned long long kLzWaitNs = 1000000000ull;   // an mbarrier wait gives up after 1 s

// meta layout: [0] M, [1] overflow (M > mcap), [2] E (terms of the step),
// [3] C (terms per thread).
constexpr int kLzMetaSize = 4;

// The equilibrium sum of entry k of the 30 from the axis sums E_p = sum A v^p (the
// three axes are alike).
__host__ __device__ inline double lz_equilibrium(int k, const double (&E)[5])
{
    const double z = E[0], e22 = E[2] * E[2] * z, e31 = E[3] * E[1] * z, e112 = E[1] * E[1] * E[2];
    double x = z * z * z;                                         // 1
    if (k >= 1 && k <= 3) x = E[1] * z * z;                       // v_i
    if (k >= 4 && k <= 6) x = E[2] * z * z;                       // v_i^2
    if (k >= 7 && k <= 9) x = E[1] * E[1] * z;                    // v_i v_j
    if (k >= 10 && k <= 12) x = E[3] * z * z;                     // v_i^3
    if (k >= 13 && k <= 18) x = E[2] * E[1] * z;                  // v_i^2 v_j
    if (k == 19) x = E[1] * E[1] * E[1];                          // v_x v_y v_z
    if (k >= 20 && k <= 22) x = E[4] * z * z + 2.0 * e22;         // v_i^2 v^2
    if (k >= 23 && k <= 25) x = 2.0 * e31 + e112;                 // v_i v_j v^2
    if (k == 26) x = 3.0 * E[2] * z * z;                          // v^2
    if (k >= 27) x = E[3] * z * z + 2.0 * E[1] * E[2] * z;        // v_i v^2
    return x;
}

// Nodes per streaming thread and stage: four consecutive jz (16-byte loads
// and stores), or two where rows of N nodes are not multiples of 16 bytes
// (N = 2 mod 4; before, such grids ran the generic per-cell kernel: ten steps of
// 192^2 x 18^3, stretched, 8192 samples, 45.4 -> 17.2 ms).
__host__ __device__ constexpr int lz_vec(int N) { return N % 4 == 0 ? 4 : 2; }

// Planes per streaming stage: the largest divisor K of N/2 with K N^2/VW <=
// ST (one node vector per streaming thread; stages never straddle jx =
// N/2, so the upwind x source is the same cell for the whole stage).  0:
// unsupported.
__host__ __device__ constexpr int lz_planes(int N, int ST)
{
    int K = 0;
    for (int k = 1; k <= N / 2; ++k)
        if ((N / 2) % k == 0 && k * (N * N / lz_vec(N)) <= ST) K = k;
    return K;
}

// Streaming threads for N nodes per axis: 512 where that raises the busy
// share by more than 1.4 (above), or where a plane needs them, else 256.
__host__ __device__ constexpr int lz_stream_threads(int N)
{
    const int s2 = lz_planes(N, 256), s5 = lz_planes(N, 512);
    return s2 == 0 || 10 * s5 * 256 > 14 * s2 * 512 ? 512 : 256;
}

// ---------------------------------------------------------------------
// Per-step plan (once per step; every cell shares it)
// ---------------------------------------------------------------------

// Marks every node a sample of the step maps to.
static __global__ void k_lz_mark(int nt, const int4 *__restrict__ idx, int *__restrict__ flag)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nt) return;
    const int4 q = idx[l];
    if (q.x >= 0) flag[q.x] = 1;
    if (q.y >= 0) flag[q.y] = 1;
    if (q.z >= 0) flag[q.z] = 1;
    if (q.w >= 0) flag[q.w] = 1;
}

// The nodes that the sample sets of steps 0, 1, ... map to, step blockIdx.y as bit
// blockIdx.y of flag, and their numbers per step (the flags cleared again): the
// compact arrays are sized by a few steps, in two launches and one read.
static __global__ void k_lz_probe(Geo g, int *__restrict__ flag)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= g.nt) return;
    const SampleOut o = draw_sample_cell<float>(g, blockIdx.y, 0xFFFFFFFFu, (uint32_t)l);
#pragma unroll
    for (int r = 0; r < 4; ++r)
        if (o.idx[r] >= 0) atomicOr(flag + o.idx[r], 1 << blockIdx.y);
}
static __global__ void k_lz_probe_count(int nvt, int *__restrict__ flag, int steps, int *__restrict__ out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int f = j < nvt ? flag[j] : 0;
    if (j < nvt) flag[j] = 0;
    for (int s = 0; s < steps; ++s) {
        const int n = __syncthreads_count(f >> s & 1);
        if (threadIdx.x == 0 && n) atomicAdd(out + s, n);
    }
}

// Compact numbering of the marked nodes (ascending node order), one CTA of
// 1024 threads: cidx[j] = m, act[m] = j, the bit mask of marked nodes and, per
// 32-node word, the compact index of its first marked node.  Clears the flags.
// Each warp forms 32 mask words from coalesced flag loads (one ballot per
// word), lane k keeping word k; warp and block scans of the word counts
// give the compact indices.
// stats (nullable): [5] counts steps whose active set exceeded mcap.
__device__ __forceinline__ void lz_scan_block(int nvt, int mcap, int *__restrict__ flag, int *__restrict__ cidx,
                                              int *__restrict__ act, uint32_t *__restrict__ mask,
                                              int *__restrict__ wpre, int *__restrict__ meta,
                                              unsigned long long *__restrict__ stats)
{
    __shared__ int wsum[32];
    __shared__ int btot;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5, nw = (nvt + 31) / 32;
    int carry = 0;
    for (int b0 = 0; b0 < nw; b0 += 1024) {
        const int base = b0 + wp * 32;                // this warp's 32 words
        uint32_t bits = 0;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const int w = base + k;
            const bool set = w * 32 + lane < nvt && flag[w * 32 + lane] != 0;
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, set);
            if (lane == k) bits = bal;
        }
        const int w = base + lane, cnt = __popc(bits);
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) wsum[wp] = inc;
        __syncthreads();
        if (wp == 0) {
            const int x0 = wsum[lane];
            int x = x0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) x += v;
            }
            wsum[lane] = x - x0;
            if (lane == 31) btot = x;
        }
        __syncthreads();
        int run = carry + wsum[wp] + inc - cnt;
        carry += btot;
        __syncthreads();                              // wsum and btot are reused
        if (w < nw) {
            mask[w] = bits;
            wpre[w] = run;
            for (uint32_t bb = bits; bb; bb &= bb - 1) {
                const int j = w * 32 + __ffs(bb) - 1;
                cidx[j] = run;
                act[run] = j;
                flag[j] = 0;
                ++run;
            }
        }
    }
    if (t == 0) {
        meta[0] = carry;
        meta[1] = carry > mcap ? 1 : 0;
        if (stats) {
            if (carry > mcap) atomicAdd(stats + 5, 1ull);
            stats[6] = (unsigned long long)carry;
        }
    }
}
static __global__ void __launch_bounds__(1024) k_lz_scan(int nvt, int mcap, int *__restrict__ flag,
                                                 int *__restrict__ cidx, int *__restrict__ act,
                                                 uint32_t *__restrict__ mask, int *__restrict__ wpre,
                                                 int *__restrict__ meta,
                                                 unsigned long long *__restrict__ stats = nullptr)
{
    lz_scan_block(nvt, mcap, flag, cidx, act, mask, wpre, meta, stats);
}

// Compact node indices (a, b, a*, b*) of every sample, and the number of
// terms per destination.
__device__ __forceinline__ void lz_remap_one(int l, const int4 *__restrict__ idx, const int *__restrict__ cidx,
                                             ushort4 *__restrict__ qc, int *__restrict__ count)
{
    const int4 q = idx[l];
    const int d[4] = {q.x >= 0 ? cidx[q.x] : -1, q.y >= 0 ? cidx[q.y] : -1,
                      q.z >= 0 ? cidx[q.z] : -1, q.w >= 0 ? cidx[q.w] : -1};
    qc[l] = Idx4<uint16_t>::make(d);
#pragma unroll
    for (int r = 0; r < 4; ++r)
        if (d[r] >= 0) atomicAdd(count + d[r], 1);
}
static __global__ void k_lz_remap(int nt, const int4 *__restrict__ idx, const int *__restrict__ cidx,
                           ushort4 *__restrict__ qc, int *__restrict__ count)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < nt) lz_remap_one(l, idx, cidx, qc, count);
}

// Exclusive scan of the term counts over the M destinations (cursor = first
// position of each destination's terms in the sorted order, rowend = one past
// its last), the number of terms E and the run length C of each of the
// kernel's T threads; clears the counts.  A destination without terms gets
// one term of weight 0 (at the zero entry M, entries of 1 << osh bytes), so
// that every destination has a row and a run steps to the next destination
// at each row end.  One CTA of 1024 threads.
__device__ __forceinline__ void lz_lscan_block(int T, int osh, int *__restrict__ count, int *__restrict__ cursor,
                                               int *__restrict__ rowend, int *__restrict__ meta,
                                               uint2 *__restrict__ rec, int *__restrict__ dest0)
{
    __shared__ int part[1024];
    const int t = threadIdx.x, M = meta[0], per = (M + 1023) / 1024;
    const int b = min(M, t * per), e = min(M, b + per);
    int s = 0;
    for (int i = b; i < e; ++i) s += max(count[i], 1);
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int v = t >= off ? part[t - off] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    // Runs of C terms, C a multiple of 8; the positions past the last term
    // hold zero records (weight 0, no destination change) and every run
    // starts at the zero entry M until k_lz_lfill names its first term.
    const int E = part[1023], C = ((E + T - 1) / T + 7) / 8 * 8;
    for (int p = E + t; p < C * T; p += 1024) {
        const int tt = p / C, i = p - tt * C;
        rec[(int64_t)i * T + tt] = make_uint2(0u, 0u);
    }
    for (int tt = t; tt < T; tt += 1024) dest0[tt] = M;
    __syncthreads();
    const uint32_t zo = (uint32_t)M << osh;
    int run = part[t] - s;
    for (int i = b; i < e; ++i) {
        cursor[i] = run;
        if (count[i] == 0) {
            const int tt = run / C, j = run - tt * C;
            rec[(int64_t)j * T + tt] = make_uint2(zo | (zo << 16) | 1u, 0u);
            if (j == 0) dest0[tt] = i;
            ++run;
        }
        run += count[i];
        rowend[i] = run;
        count[i] = 0;
    }
    if (t == 1023) {
        meta[2] = E;
        meta[3] = C;
    }
}
static __global__ void __launch_bounds__(1024) k_lz_lscan(int T, int osh, int *__restrict__ count,
                                                         int *__restrict__ cursor,
                                                         int *__restrict__ rowend,
                                                         int *__restrict__ meta, uint2 *__restrict__ rec,
                                                         int *__restrict__ dest0)
{
    lz_lscan_block(T, osh, count, cursor, rowend, meta, rec, dest0);
}

// The term records, sorted by destination: position p of the sorted order
// goes to thread p / C, slot i = p mod C, stored at rec[i T + p / C] so that
// the threads' i-th records are adjacent.  A record is
//   x = a_off | b_off << 16 | last,   y = +-W (bits of the float),
// with a_off, b_off the byte offsets of the sample's pre-collision nodes in
// the kernel's compact array (entries of 1 << osh bytes; a node outside the
// grid points to the zero entry M), last set on the final term of a
// destination, and the sign negative for the loss terms (the destination is
// a or b).  dest0[tt] is the destination of thread tt's first term.
// Nothing is written when the step overflowed (the kernel does not run then).
template <typename PA>
__device__ __forceinline__ void lz_lfill_one(int l, int T, int osh, const ushort4 *__restrict__ qc,
                                             const PA *__restrict__ pa, int *__restrict__ cursor,
                                             const int *__restrict__ rowend, const int *__restrict__ meta,
                                             uint2 *__restrict__ rec, int *__restrict__ dest0)
{
    if (meta[1]) return;
    const int M = meta[0], C = meta[3];
    const ushort4 q = qc[l];
    const int d[4] = {idx_of(q.x), idx_of(q.y), idx_of(q.z), idx_of(q.w)};
    const uint32_t ao = (uint32_t)(d[0] >= 0 ? d[0] : M) << osh;
    const uint32_t bo = (uint32_t)(d[1] >= 0 ? d[1] : M) << osh;
    const uint32_t x = ao | (bo << 16);
    const float W = pa[l].W;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (d[r] < 0) continue;
        const int pos = atomicAdd(cursor + d[r], 1);
        const int tt = pos / C, i = pos - tt * C;
        const uint32_t last = pos == rowend[d[r]] - 1 ? 1u : 0u;
        rec[(int64_t)i * T + tt] = make_uint2(x | last, __float_as_uint(r < 2 ? -W : W));
        if (i == 0) dest0[tt] = d[r];
    }
}
template <typename PA>
__global__ void k_lz_lfill(int nt, int T, int osh, const ushort4 *__restrict__ qc,
                           const PA *__restrict__ pa, int *__restrict__ cursor,
                           const int *__restrict__ rowend, const int *__restrict__ meta,
                           uint2 *__restrict__ rec, int *__restrict__ dest0)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < nt) lz_lfill_one(l, T, osh, qc, pa, cursor, rowend, meta, rec, dest0);
}

// Bank-aware order of the term records.  A collision thread reads the two
// operands of its term with two 16-byte (G = 4) or 8-byte (G = 2) shared
// loads.  The loads of a warp are served NB = 8 (or 16) lanes at a time, one
// wavefront per distinct entry in the busiest of the NB bank groups (entry
// index mod NB), so the NB runs that one phase reads together are ordered
// jointly.  Terms move only inside their destination segment of a run, and
// the two operands of a term may be swapped (the product is symmetric).
// Position by position, the runs choose in order of how few choices they
// have left (the one with the fewest remaining terms in its segment first;
// padding, which reads entry 0, before all): each takes the remaining term
// of its segment, and the operand order, whose first and second operands
// meet the fewest bank groups already holding another entry at that
// position.  A run decides position p once it has decided p - 1 and every
// run before it at p has decided p.  The positions are cut into chunks
// ordered independently (a segment that crosses a chunk's end is cut
// there).  One warp per phase group and chunk: NB runs x 32 / NB lanes that
// scan a run's choices.  Nothing happens if a run is longer than cmax.
// Several plans at once: blockIdx.z selects plan slot (z0 + blockIdx.z) mod
// zK, whose meta and records lie kLzMetaSize ints and rec_stride records
// after those of slot 0.
constexpr int kLzOrderWin = 64;     // positions whose taken entries are held at a time

__host__ __device__ inline size_t lz_order_smem(int chunk, int nb)
{
    // records (rows padded to an odd length), taken entries of a window of
    // positions, segment ends, run order masks, decided masks of the window,
    // padding masks
    const size_t m = nb == 8 ? 1 : 2;
    return (size_t)nb * (chunk + 1) * sizeof(uint2) + (size_t)kLzOrderWin * nb * sizeof(uint32_t) +
           (size_t)chunk * nb * (sizeof(uint16_t) + m) + (size_t)kLzOrderWin * m + (size_t)chunk * m + 32;
}

template <int NB>
__global__ void __launch_bounds__(32) k_lz_order(int T, int cmax, int chunk, const int *__restrict__ meta,
                                                 uint2 *__restrict__ rec, int zK = 1, int z0 = 0,
                                                 int64_t rec_stride = 0)
{
    {
        const int zs = (z0 + (int)blockIdx.z) % zK;
        meta += zs * kLzMetaSize;
        rec += zs * rec_stride;
    }
    static_assert(NB == 8 || NB == 16, "phase width");
    constexpr int H = 32 / NB;                       // lanes per run
    constexpr int OSH = NB == 8 ? 4 : 3;             // log2 of the entry size
    constexpr int W = kLzOrderWin;
    constexpr uint16_t kNone = 0xFFFF;
    using Mask = typename std::conditional<NB == 8, uint8_t, uint16_t>::type;
    extern __shared__ __align__(16) unsigned char osm[];
    const int lane = threadIdx.x, l = lane / H, h = lane - l * H;
    const unsigned rmask = ((1u << H) - 1u) << (l * H);   // the lanes of this run
    const int tt = blockIdx.x * NB + l;
    const int C = meta[3], c0 = blockIdx.y * chunk;
    if (C > cmax || meta[1] || blockIdx.x * NB + NB > T || c0 >= C) return;
    const int L = min(chunk, C - c0), SP = chunk + 1;
    uint2 *b = reinterpret_cast<uint2 *>(osm);                   // [NB][SP] working copies of the runs
    uint32_t *u = reinterpret_cast<uint32_t *>(b + NB * SP);     // [W][NB] entries taken: first | second << 16
    uint16_t *seg = reinterpret_cast<uint16_t *>(u + W * NB);    // [NB][chunk] segment end | last << 15
    Mask *bm = reinterpret_cast<Mask *>(seg + NB * chunk);       // [NB][chunk] runs that choose before this one
    Mask *dec = bm + NB * chunk;                                // [W] runs that have decided p
    Mask *pad = dec + W;                                        // [chunk] runs that are padding at p
    // Positions p live in slot p mod W of u and dec while some run has not
    // decided them; a run decides p only while p < (the smallest undecided
    // position) + W, which delays some decisions but changes none.
#pragma unroll 4
    for (int i = lane; i < NB * L; i += 32) {       // the NB runs of a position are adjacent in rec
        const int p = i / NB, r = i - p * NB;
        b[r * SP + p] = rec[(int64_t)(c0 + p) * T + blockIdx.x * NB + r];
    }
    __syncwarp();
    // Segments: up to a destination's last term or the chunk's end, before
    // the padding (zero records).
    if (h == 0) {
        const uint2 *br = b + l * SP;
        uint16_t *se = seg + l * chunk;
        int i = 0;
        while (i < L && !(br[i].x == 0u && br[i].y == 0u)) {
            int e = i;                                // the segment's last position (< L)
            while (e + 1 < L && !(br[e].x & 1u) && !(br[e + 1].x == 0u && br[e + 1].y == 0u)) ++e;
            const uint16_t v = (uint16_t)(e | (br[e].x & 1u) << 15);
            for (int p = i; p <= e; ++p) se[p] = v;
            i = e + 1;
        }
        for (int p = i; p < L; ++p) se[p] = kNone;
    }
    __syncwarp();
    // Per position: the order of the runs (remaining choices, then run
    // index); padding is decided from the start and reads entry 0.
    for (int p = lane; p < L; p += 32) {
        int sz[NB];
        Mask d = 0;
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const uint16_t v = seg[r * chunk + p];
            sz[r] = v == kNone ? 0 : (v & 0x7FFF) - p + 1;
            if (v == kNone) d |= (Mask)(1u << r);
        }
        pad[p] = d;
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            Mask m = 0;
#pragma unroll
            for (int r2 = 0; r2 < NB; ++r2)
                if (sz[r2] < sz[r] || (sz[r2] == sz[r] && r2 < r)) m |= (Mask)(1u << r2);
            bm[r * chunk + p] = m;
        }
    }
    __syncwarp();
    // The first window: nothing taken, padding decided (its reads are entry 0).
    int wend = min(W, L);                             // positions below this hold their slot
    for (int i = lane; i < wend * NB; i += 32) {
        const int q = i / NB, g = i - q * NB;
        u[i] = g == 0 && pad[q] ? 0u : 0xFFFFFFFFu;
    }
    for (int q = lane; q < wend; q += 32) dec[q] = pad[q];
    __syncwarp();
    uint2 *bl = b + l * SP;
    const uint16_t *sl = seg + l * chunk;
    const Mask *bml = bm + l * chunk;
    int p = 0;                                        // this run's next position in the chunk
    uint16_t sv = L > 0 ? sl[0] : kNone;              // its segment: end | last << 15, kNone: padding
    // Every step some run is ready (the first, at the smallest undecided
    // position, in that position's order; that position lies in the window),
    // so NB * L steps always suffice.
    for (int step = 0; step < NB * L; ++step) {
        const bool active = p < L && sv != kNone;
        if (!__any_sync(0xFFFFFFFFu, active)) break;
        // The smallest undecided position; positions up to it + W get slots.
        const int pmin = (int)__reduce_min_sync(0xFFFFFFFFu, (unsigned)(active ? p : L));
        const int wnew = min(pmin + W, L);
        if (wnew > wend) {
            // (positions below wnew - W are behind every run: not set up)
            const int w0 = max(wend, wnew - W);
            for (int i = lane; i < (wnew - w0) * NB; i += 32) {
                const int q = w0 + i / NB, g = i % NB;
                u[(q & (W - 1)) * NB + g] = g == 0 && pad[q] ? 0u : 0xFFFFFFFFu;
            }
            for (int q = w0 + lane; q < wnew; q += 32) dec[q & (W - 1)] = pad[q];
            wend = wnew;
            __syncwarp();
        }
        bool ready = false;
        Mask dp = 0;
        if (active && p < wend) {
            const Mask need = bml[p];
            dp = dec[p & (W - 1)];
            ready = (Mask)(dp & need) == need;
        }
        __syncwarp();                                 // the reads above precede this step's writes
        uint32_t best = 0xFFFFFFFFu;                  // cost << 24 | swap << 23 | position
        const int s1 = sv & 0x7FFF;
        const uint32_t *row = u + (p & (W - 1)) * NB; // entries taken at p, by group
        if (ready) {
            // Passes of 4 H candidates; the run's lanes take the same passes.
            for (int jb = p; jb <= s1; jb += 4 * H) {
                const int j0 = jb + h;
                uint32_t xs[4], wa[4], wb[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) xs[k] = j0 + k * H <= s1 ? bl[j0 + k * H].x : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    wa[k] = row[(xs[k] >> OSH) & (NB - 1)];
                    wb[k] = row[(xs[k] >> (16 + OSH)) & (NB - 1)];
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = j0 + k * H;
                    if (j > s1) break;
                    const uint32_t ea = (xs[k] & 0xFFFCu) >> OSH, eb = xs[k] >> (16 + OSH);
                    const uint32_t a1 = wa[k] & 0xFFFFu, a2 = wa[k] >> 16, b1 = wb[k] & 0xFFFFu, b2 = wb[k] >> 16;
                    const uint32_t cn = (a1 != kNone && a1 != ea) + (b2 != kNone && b2 != eb);
                    const uint32_t cs = (b1 != kNone && b1 != eb) + (a2 != kNone && a2 != ea);
                    const uint32_t key = cs < cn ? (cs << 24 | 1u << 23 | (uint32_t)j) : (cn << 24 | (uint32_t)j);
                    best = min(best, key);
                }
                // A candidate with no conflict and no swap beats every later
                // one (the key then orders by position): the scan stops.
#pragma unroll
                for (int o = 1; o < H; o <<= 1) best = min(best, __shfl_xor_sync(rmask, best, o));
                if (best < (1u << 23)) break;
            }
        }
#pragma unroll
        for (int o = 1; o < H; o <<= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
        if (ready && h == 0) {
            const int j = (int)(best & 0xFFFFu);
            uint2 r = bl[j];
            const uint2 front = bl[p];
            r.x &= ~1u;
            if (best >> 23 & 1u) r.x = (r.x >> 16) | ((r.x & 0xFFFCu) << 16);
            if (p == s1) r.x |= (uint32_t)(sv >> 15);
            rec[(int64_t)(c0 + p) * T + tt] = r;
            bl[j] = front;                            // the front term fills the hole
            const uint32_t e1 = (r.x & 0xFFFCu) >> OSH, e2 = r.x >> (16 + OSH);
            const uint32_t g1 = e1 & (NB - 1), g2 = e2 & (NB - 1);
            uint32_t v1 = row[g1];
            if ((v1 & 0xFFFFu) == kNone) v1 = (v1 & 0xFFFF0000u) | e1;
            uint32_t v2 = g2 == g1 ? v1 : row[g2];
            if ((v2 >> 16) == kNone) v2 = (v2 & 0xFFFFu) | e2 << 16;
            uint32_t *roww = u + (p & (W - 1)) * NB;
            roww[g1] = g2 == g1 ? v2 : v1;
            if (g2 != g1) roww[g2] = v2;
            dec[p & (W - 1)] = (Mask)(dp | (1u << l));
        }
        __syncwarp();
        if (ready) {
            ++p;
            if (p > s1) sv = p < L ? sl[p] : kNone;
        }
    }
    // Positions left undecided (none when the loop ran out normally) keep
    // their remaining terms, with the destination bit at the segment end.
    if (h == 0)
        for (; p < L && sl[p] != kNone; ++p) {
            uint2 r = bl[p];
            r.x &= ~1u;
            if (p == (sl[p] & 0x7FFF)) r.x |= (uint32_t)(sl[p] >> 15);
            rec[(int64_t)(c0 + p) * T + tt] = r;
        }
}

// ---------------------------------------------------------------------
// Fallback when a step has more active nodes than mcap: the k_cell4 plan (or,
// for N = 2 mod 4, that of the generic kernel, in logical node order) is
// derived from the logical one, the input is corrected in place and mu_out
// is cleared (those kernels write corrected states).  All return at once
// otherwise.
// ---------------------------------------------------------------------
__device__ __forceinline__ void lz_fb_plan_one(int l, int N, const int4 *__restrict__ idx,
                                               const PlanA<float, int> *__restrict__ pa,
                                               ushort4 *__restrict__ pidx16, PlanA<float, uint16_t> *__restrict__ pa16,
                                               int *__restrict__ count)
{
    const int4 q = idx[l];
    int o[4] = {q.x, q.y, q.z, q.w};
    const int nq = N / 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int j = o[k];
        if (j < 0 || N % 4 != 0) continue;
        const int jx = j / (N * N), jz = j % N, row = j - jz;
        int r = jz / 4 + jx % nq;
        if (r >= nq) r -= nq;
        o[k] = row + 4 * r + (jz & 3);
    }
    const ushort4 u = Idx4<uint16_t>::make(o);
    pidx16[l] = u;
    pa16[l] = make_plan_a<float, uint16_t>(o[0], o[1], (double)pa[l].W);
    if (!count) return;
    if (u.x != 0xFFFF) atomicAdd(count + u.x, 1);
    if (u.y != 0xFFFF) atomicAdd(count + u.y, 1);
    if (u.z != 0xFFFF) atomicAdd(count + u.z, 1);
    if (u.w != 0xFFFF) atomicAdd(count + u.w, 1);
}
static __global__ void k_lz_fb_plan(int nt, int N, const int *__restrict__ meta,
                             const int4 *__restrict__ idx, const PlanA<float, int> *__restrict__ pa,
                             ushort4 *__restrict__ pidx16, PlanA<float, uint16_t> *__restrict__ pa16,
                             int *__restrict__ count)
{
    if (!meta[1]) return;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < nt) lz_fb_plan_one(l, N, idx, pa, pidx16, pa16, count);
}

// h <- h_c + (1 + eps h_c)(mu_c . psi_j) for every node (in place allowed:
// hout may be hin, so neither is restrict-qualified); mu_zero (nullable) is
// then cleared, and mu_used (nullable; may be mu) gets each cell's
// corrections cleared once they are read.  When skip_unless (nullable)
// points to 0, does nothing.  One CTA per cell at a time; float4 over jz.
static __global__ void k_lz_materialize(Geo g, const int *__restrict__ skip_unless,
                                 const float *hin, const float *mu, float *hout,
                                 float *__restrict__ mu_zero, float *mu_used = nullptr)
{
    if (skip_unless && !skip_unless[1]) return;
    __shared__ float sv[kMaxN];
    __shared__ float smu[8];
    const int N = g.nv, nq = N / 4, Q = N * N / 4;
    const bool rows4 = N % 4 == 0;                   // a float4 lies in one row
    for (int i = threadIdx.x; i < N; i += blockDim.x) sv[i] = (float)g.axv[i];
    const float eps = g.epsf;
    const int64_t plane = g.nvt / 4;
    for (int c = blockIdx.x; c < g.nr; c += gridDim.x) {
        __syncthreads();
        if (threadIdx.x < 8) smu[threadIdx.x] = mu[(int64_t)c * 8 + threadIdx.x];
        __syncthreads();
        if (mu_used && threadIdx.x < 8) mu_used[(int64_t)c * 8 + threadIdx.x] = 0.f;
        const float4 *src = reinterpret_cast<const float4 *>(hin) + (int64_t)c * plane;
        float4 *dst = reinterpret_cast<float4 *>(hout) + (int64_t)c * plane;
        for (int o = threadIdx.x; o < (int)plane; o += blockDim.x) {
            float4 h = src[o];
            float *hp = &h.x;
            if (rows4) {
                const int jx = o / Q, q = o % Q, jy = q / nq, jz = 4 * (q % nq);
                const float vx = sv[jx], vy = sv[jy];
#pragma unroll
                for (int i = 0; i < 4; ++i) hp[i] = state_corr(hp[i], state_kappa(smu, vx, vy, sv[jz + i]), eps);
            } else {
#pragma unroll
                for (int i = 0; i < 4; i += 2) {     // (two nodes of a row)
                    const int j = 4 * o + i, jxy = j / N, jx = jxy / N, jz = j - jxy * N;
                    const float vx = sv[jx], vy = sv[jxy - jx * N];
                    hp[i] = state_corr(hp[i], state_kappa(smu, vx, vy, sv[jz]), eps);
                    hp[i + 1] = state_corr(hp[i + 1], state_kappa(smu, vx, vy, sv[jz + 1]), eps);
                }
            }
            dst[o] = h;
        }
    }
    if (mu_zero) {
        const int64_t n = (int64_t)g.nr * 8;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x)
            mu_zero[i] = 0.f;
    }
}

// ---------------------------------------------------------------------
// Packed FP32x2 arithmetic (each component rounds like fmaf / __fadd_rn).
// ---------------------------------------------------------------------
__device__ __forceinline__ float2 lz_add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 lz_mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 lz_fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 lz_dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 lz_lo(float4 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float2 lz_hi(float4 a) { return make_float2(a.z, a.w); }

// Values of a node in the G cells of a group (adjacent in shared memory).
template <int G> struct LzVec;
template <> struct LzVec<2> { using T = float2; };
template <> struct LzVec<4> { using T = float4; };

__device__ __forceinline__ float2 lz_zero2() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ void lz_set_zero(float2 &a) { a = lz_zero2(); }
__device__ __forceinline__ void lz_set_zero(float4 &a) { a = make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ void lz_atomic_add(float2 *p, float2 v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
__device__ __forceinline__ void lz_atomic_add(float4 *p, float4 v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
    atomicAdd(&p->z, v.z);
    atomicAdd(&p->w, v.w);
}

// ---------------------------------------------------------------------
// Per-thread asynchronous copies global -> shared (cp.async), completed by
// the issuing thread's cp.async.wait_group: each thread prefetches the source
// values of its own nodes several streaming stages ahead, with no register
// cost and no synchronisation with other threads.
// ---------------------------------------------------------------------
__device__ __forceinline__ uint32_t lz_saddr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lz_cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(lz_saddr(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void lz_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void lz_cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// All but the newest n (1 .. kLzMaxStages - 1) groups of this thread's copies
// have landed.
__device__ __forceinline__ void lz_cp_wait_but(int n)
{
    if (n >= 4) asm volatile("cp.async.wait_group 4;" ::: "memory");
    else if (n == 3) asm volatile("cp.async.wait_group 3;" ::: "memory");
    else if (n == 2) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else asm volatile("cp.async.wait_group 1;" ::: "memory");
}

// Bulk copies global -> shared through the tensor-memory-access unit
// (cp.async.bulk, completion counted in bytes on an mbarrier) and the
// mbarrier operations of the streaming ring.  Every wait is bounded: each
// poll returns within the hardware's own suspend limit, and after kLzWaitNs
// of the global timer the wait gives up and returns false.
__device__ __forceinline__ void lz_mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void lz_mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void lz_mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void lz_mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool lz_mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long lz_now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool lz_mbar_wait(uint32_t bar, uint32_t parity)
{
    if (lz_mbar_try(bar, parity)) return true;
    const unsigned long long t0 = lz_now_ns();
    while (!lz_mbar_try(bar, parity))
        if (lz_now_ns() - t0 > kLzWaitNs) return false;
    return true;
}
// A bounded wait that is skipped once any wait of the CTA has given up (the
// CTA then finishes without waiting and reports the error).
__device__ __forceinline__ void lz_ring_wait(uint32_t bar, uint32_t parity, int &err)
{
    volatile int *e = &err;
    if (*e == 0 && !lz_mbar_wait(bar, parity)) *e = 1;
}
__device__ __forceinline__ void lz_bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Orders this thread's generic-proxy shared-memory writes before later
// bulk copies (async proxy) into the same bytes.
__device__ __forceinline__ void lz_fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Everything the kernel needs besides the geometry (by value).
struct LzArgs {
    const float *hin, *mu_in, *ghost;
    float *hout, *mu_out;
    double *mom;
    const uint2 *rec;       // term records (k_lz_lfill)
    const int *dest0;       // first destination of each thread's run
    const int *meta;
    const uint32_t *mask;
    const int *wpre, *act;
    int mcap;
    float e0[kLzX];         // sum_j w_j X_k(v_j) of the 30 monomials
    long long *clk;         // nullable: phase trace of CTA 0 (kClkCells groups x kClkPhases)
    unsigned long long *stats;  // nullable: [3] counts correction solves that fell back
    int nostream;           // 1: h~ = h (no free streaming; the relaxation alone)
    int early_tail;         // 1: the collision warps start the increment sums at once
    unsigned long long *err;    // nullable: set to 1 when a bounded mbarrier wait gave up
    int tx_excess;          // bulk-copy ring, CTA 0's first stage: bytes expected beyond
                            // those copied (a wait that runs out, for tests; normally 0)
    int *fb_count;          // nullable: counts of the fallback's scatter list, zeroed
    int fb_n;               // (fb_n ints) when the step overflowed, before the fallback
    int stages;             // streaming stages held in shared memory
};

// Shared memory.  A fixed-layout head (compile-time offsets): warp partial
// sums, per-axis tables, the groups' cells and the correction tables of the
// cells the streaming reads.  Then two compact arrays of h~ (G values per
// active node plus a zero entry; the streaming warps fill one while the
// collision warps use the other), the compact array of collision
// increments, the per-thread staging slots of the streaming prefetch
// (the stages x {own, x source, y source} x streaming threads, 16 bytes
// each), the active-node bit mask, its word prefixes and the node list.
struct alignas(128) LzHead {
    float fpart[kLzMaxG][kLzMaxStreamT / 32][32];    // warp partials of the F sums
    float ftot[3][kLzMaxG][2][32];               // their totals (sum, error), per group (it mod 3)
    float dpart[2][kLzMaxG][kLzDParts][32];      // partials of the D sums, per group (it mod 2)
    float4 ta[kLzMaxN];                          // -ax, -ax, A, A
    float4 tv12[kLzMaxN];                        // v, v, v^2, v^2
    float4 tv34[kLzMaxN];                        // v^3, v^3, v^4, v^4
    float v[kLzMaxN], A[kLzMaxN], IA[kLzMaxN], cuy[kLzMaxN];
    float4 tcx[kLzMaxG][kLzMaxN];                // ca of the own and the upwind x cell, duplicated
    float2 tcy[kLzMaxG][2][kLzMaxN];             // ca of the cell below (0) and above (1), duplicated
    float mus[kLzMaxG][5][8];                    // mu of own, right, left, below, above (0 outside)
    int4 cell[2][kLzMaxG];                       // c, ix, iy of a group's cells (c < 0: none), per buffer
    float e0[32];                                // equilibrium sums of the 30 monomials
    unsigned char px[5][16];                     // lz_psiphi
    int tail_next;                               // next chunk of the increment sums to claim
    int tma_err;                                 // a bounded wait of the bulk-copy ring gave up
    unsigned long long bar_full[kLzMaxStages];      // bulk-copy ring: stage landed (transaction bytes)
    unsigned long long bar_empty[kLzMaxStages];     // bulk-copy ring: stage read by the streaming warps
};
constexpr uint32_t kLzAOff = (sizeof(LzHead) + 15) & ~(size_t)15;

struct LzOff {
    uint32_t abytes, a1, bc, ring, mask, act, end;
};
__host__ __device__ inline LzOff lz_offsets(int nvt, int mcap, int G, int stages, int S, int VW)
{
    LzOff o;
    o.abytes = (uint32_t)(((sizeof(float) * (size_t)G * (mcap + 1)) + 127) & ~(size_t)127);
    size_t off = kLzAOff + o.abytes;
    o.a1 = (uint32_t)off; off += o.abytes;
    o.bc = (uint32_t)off; off += o.abytes;
    o.ring = (uint32_t)off; off += (size_t)stages * 3 * S * VW * sizeof(float);
    o.mask = (uint32_t)off; off += sizeof(uint2) * ((nvt + 31) / 32);
    o.act = (uint32_t)off; off += sizeof(uint16_t) * (size_t)mcap;
    o.end = (uint32_t)((off + 15) & ~(size_t)15);
    return o;
}

// Monomial index of psi_a * phi_b in the 30-entry sum vector X (psi = 1,
// v_x, v_y, v_z, v^2; phi = 1, v_x, v_y, v_z, v_x^2, v_y^2, v_z^2, v_x v_y,
// v_x v_z, v_y v_z).  X order: 0 1; 1-3 v_x, v_y, v_z; 4-6 v_x^2, v_y^2,
// v_z^2; 7-9 v_x v_y, v_x v_z, v_y v_z; 10-12 v_x^3, v_y^3, v_z^3; 13 v_x^2 v_y;
// 14 v_x^2 v_z; 15 v_x v_y^2; 16 v_y^2 v_z; 17 v_x v_z^2; 18 v_y v_z^2;
// 19 v_x v_y v_z; 20-22 v_x^2 v^2, v_y^2 v^2, v_z^2 v^2; 23-25 v_x v_y v^2,
// v_x v_z v^2, v_y v_z v^2; 26 v^2; 27-29 v_x v^2, v_y v^2, v_z v^2.
__host__ __device__ constexpr int lz_psiphi(int a, int b)
{
    constexpr unsigned char t[5][10] = {
        {0, 1, 2, 3, 4, 5, 6, 7, 8, 9},
        {1, 4, 7, 8, 10, 15, 17, 13, 14, 19},
        {2, 7, 5, 9, 13, 11, 18, 15, 19, 16},
        {3, 8, 9, 6, 14, 16, 12, 19, 17, 18},
        {26, 27, 28, 29, 20, 21, 22, 23, 24, 25}};
    return t[a][b];
}

// The 26 monomial sums of sum_nodes n(v) from per-thread power sums over jx
// (s[p] = sum n v_x^p) at fixed v_y = y, v_z = z.
__device__ __forceinline__ void lz_mono_from_powers(const float (&s)[5], float y, float z,
                                                    float (&M)[32])
{
    const float y2 = y * y, z2 = z * z, q = y2 + z2, yz = y * z;
    M[0] += s[0];
    M[1] += s[1];
    M[2] += y * s[0];
    M[3] += z * s[0];
    M[4] += s[2];
    M[5] += y2 * s[0];
    M[6] += z2 * s[0];
    M[7] += y * s[1];
    M[8] += z * s[1];
    M[9] += yz * s[0];
    M[10] += s[3];
    M[11] += y2 * y * s[0];
    M[12] += z2 * z * s[0];
    M[13] += y * s[2];
    M[14] += z * s[2];
    M[15] += y2 * s[1];
    M[16] += y2 * z * s[0];
    M[17] += z2 * s[1];
    M[18] += y * z2 * s[0];
    M[19] += yz * s[1];
    const float t2 = s[2] + q * s[0];
    M[20] += s[4] + q * s[2];
    M[21] += y2 * t2;
    M[22] += z2 * t2;
    M[23] += y * (s[3] + q * s[1]);
    M[24] += z * (s[3] + q * s[1]);
    M[25] += yz * t2;
}

// Sum of 32 values over a warp, left with lane l holding the total of value l
// (recursive halving: 31 shuffles instead of 32 x 5).
__device__ __forceinline__ float lz_warp_reduce_scatter(float (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? v[i] : v[i + o];
            const float keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
    }
    return v[0];
}

// The pivoted fallback of a cell's 5 x 5 solve.
static __device__ __noinline__ void lz_solve_fallback_p(const Geo *g, const float *P, float *mu)
{
    double Pd[19], m8[5];
    for (int k = 0; k < 19; ++k) Pd[k] = (double)P[k];
    int f2 = 0;
    correction_solve<float>(*g, Pd, m8, &f2);
    for (int k = 0; k < 5; ++k) mu[k] = (float)m8[k];
}
__device__ __forceinline__ void lz_solve_fallback(const Geo &g, const float (&P)[19], float (&mu)[5])
{
    float p[19], m[5];                 // (copies, so that P and mu stay in registers)
#pragma unroll
    for (int k = 0; k < 19; ++k) p[k] = P[k];
    lz_solve_fallback_p(&g, p, m);
#pragma unroll
    for (int k = 0; k < 5; ++k) mu[k] = m[k];
}

// Moments of h^{n+1} (Eqs. densita..sforzi) of an FP32 cell from the sums X of N_c
// over the 30 monomials, the rounding errors Xl of the first ten, the
// equilibrium sums e0 and the correction mu: sum w h phi = sum N_c phi + sum_a
// mu_a (E0 + eps sum N_c psi_a phi).  One warp: lane b sums moment b and writes
// output b.  Every value that ends in an output is a float and its rounding error.
// (With every operation rounded to FP32 the moments after one step were 1.08e-7 off
// at 15 nodes per axis and 7.7e-8 at 30, where FP32 sums over the stored result,
// k_cell's, are 9.1e-8 and 6.0e-8 off; now 8.4e-8 and 4.6e-8, at the same time
// per step.  In FP64 the chain of about 25 operations took 5 % of a step of 192^2 x 18^3.)
__device__ __forceinline__ void lz_moments(const float *X, const float *Xl, const float *e0,
                                           const unsigned char *px, const float (&mu)[5], float eps,
                                           double *__restrict__ mom)
{
    const unsigned all = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    float m = 0.f, ml = 0.f;                           // moment b: m + ml
    if (lane < 10) {
        float d = Xl[lane];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const int x = px[k * 16 + lane];
            d = fmaf(mu[k], fmaf(eps, X[x], e0[x]), d);
        }
        two_sum(X[lane], d, m, ml);
    }
    const float rho = __shfl_sync(all, m, 0), rl = __shfl_sync(all, ml, 0);
    const float n = fmaf(eps, rho, 1.f), nl = fmaf(eps, rl, fmaf(eps, rho, 1.f - n)), in = 1.f / n;
    // (2/3) tr - rho, tr = sum of the second moments
    float tr, t1, t2, e1, b, bl;
    two_sum(__shfl_sync(all, m, 4), __shfl_sync(all, m, 5), t1, e1);
    two_sum(t1, __shfl_sync(all, m, 6), tr, t2);
    const float trl = (e1 + t2) + ((__shfl_sync(all, ml, 4) + __shfl_sync(all, ml, 5)) + __shfl_sync(all, ml, 6));
    constexpr float c = 2.f / 3.f, cl = (float)(2.0 / 3.0 - (double)c);
    const float p = c * tr, pl = fmaf(c, tr, -p) + fmaf(c, trl, cl * tr);
    two_sum(p, -rho, b, bl);
    bl += pl - rl;
    // over n: lanes 1-3 their moment, lane 4 the above
    const float h = lane == 4 ? b : m, hl = lane == 4 ? bl : ml;
    const float q = h * in, ql = (fmaf(-q, n, h) + fmaf(-q, nl, hl)) * in;
    const float u0 = __shfl_sync(all, q, 1), u1 = __shfl_sync(all, q, 2), u2 = __shfl_sync(all, q, 3);
    const float mq = __shfl_sync(all, m, lane - 1 & 31), mql = __shfl_sync(all, ml, lane - 1 & 31);
    const float ua = lane == 5 || lane == 8 || lane == 9 ? u0 : lane == 6 || lane == 10 ? u1 : u2;
    const float ub = lane == 5 ? u0 : lane == 6 || lane == 8 ? u1 : u2;
    float o = 2.f * mq, ol = fmaf(-2.f * eps * n * ua, ub, 2.f * mql);
    if (lane < 5) {
        o = lane == 0 ? m : q;
        ol = lane == 0 ? ml : ql;
    }
    if (lane == 4) ol -= c * eps * (u0 * u0 + u1 * u1 + u2 * u2);
    if (lane < 11) mom[lane] = (double)o + (double)ol;
}

// Correction and output moments of one cell from the 26 sums T (of the
// post-collision N_c = N + dN; the row has room for the 30-entry vector X), their
// rounding errors Tl and D (of the collision increment dN), all in shared memory:
// mu to mu_out, moments to mom.  Called by all 32 lanes of a warp: every lane
// solves the 5 x 5 system (the lanes share its residual), then lane b sums moment
// b and writes output b.  (With the moments summed by one lane, through arrays
// in local memory, a solve took 5-8 thousand cycles.)
__device__ __forceinline__ void lz_finish(const Geo &g, const LzArgs &a, int c, float *T, const float *Tl,
                                          const float *D, const float *e0, const unsigned char *px, int *fallback)
{
    const int lane = threadIdx.x & 31;
    if (lane >= kLzMono && lane < kLzX) {
        const int i = lane - kLzMono;            // v^2, v_x v^2, v_y v^2, v_z v^2
        T[lane] = i == 0 ? T[4] + T[5] + T[6] : i == 1 ? T[10] + T[15] + T[17]
                  : i == 2 ? T[13] + T[11] + T[18] : T[14] + T[16] + T[12];
    }
    __syncwarp();
    // Eqs. rinorm_a, correzione: G mu = -D with G from the sums of N_c and
    // D the conserved moments of the increment (1, v, v^2).
    float P[19];
#pragma unroll
    for (int k = 0; k < 10; ++k) P[k] = T[k];
    P[10] = T[27];
    P[11] = T[28];
    P[12] = T[29];
    P[13] = T[20] + T[21] + T[22];
    P[14] = D[0];
    P[15] = D[1];
    P[16] = D[2];
    P[17] = D[3];
    P[18] = D[4] + D[5] + D[6];
    float mu[5];
    if (!correction_spd(g, P, mu, lane)) {
        lz_solve_fallback(g, P, mu);
        if (lane == 0) ++*fallback;
    }
    if (lane < 5) {
        float m = mu[0];
#pragma unroll
        for (int k = 1; k < 5; ++k) m = lane == k ? mu[k] : m;
        a.mu_out[(int64_t)c * 8 + lane] = m;
    }
    if (!a.mom) return;
    lz_moments(T, Tl, e0, px, mu, g.epsf, a.mom + (int64_t)c * 11);
}

// The (v_y, v_z) part of a cell's pending correction at a thread's nodes (jy;
// jz .. jz + VW - 1): mu_y v_y + mu_z v_z + mu_4 (v_y^2 + v_z^2), as node pairs.
template <int VW>
__device__ __forceinline__ void lz_bd(const float *mu, const float *v, int jy, int jz, float2 (&bd)[VW / 2])
{
    const float vy = v[jy];
    float b[VW];
#pragma unroll
    for (int i = 0; i < VW; ++i) {
        const float vz = v[jz + i];
        b[i] = mu[2] * vy + mu[3] * vz + mu[4] * (vy * vy + vz * vz);
    }
#pragma unroll
    for (int p = 0; p < VW / 2; ++p) bd[p] = make_float2(b[2 * p], b[2 * p + 1]);
}

// lz_mono_from_powers for two cells at once (s and M hold one value per
// cell; y and z are the node's, shared by both).
__device__ __forceinline__ void lz_mono_from_powers2(const float2 (&s)[5], float y, float z,
                                                     float2 (&M)[32])
{
    const float y2 = y * y, z2 = z * z, q = y2 + z2, yz = y * z;
    const float2 Y = lz_dup(y), Z = lz_dup(z), Y2 = lz_dup(y2), Z2 = lz_dup(z2), YZ = lz_dup(yz);
    M[0] = lz_add2(M[0], s[0]);
    M[1] = lz_add2(M[1], s[1]);
    M[2] = lz_fma2(Y, s[0], M[2]);
    M[3] = lz_fma2(Z, s[0], M[3]);
    M[4] = lz_add2(M[4], s[2]);
    M[5] = lz_fma2(Y2, s[0], M[5]);
    M[6] = lz_fma2(Z2, s[0], M[6]);
    M[7] = lz_fma2(Y, s[1], M[7]);
    M[8] = lz_fma2(Z, s[1], M[8]);
    M[9] = lz_fma2(YZ, s[0], M[9]);
    M[10] = lz_add2(M[10], s[3]);
    M[11] = lz_fma2(lz_dup(y2 * y), s[0], M[11]);
    M[12] = lz_fma2(lz_dup(z2 * z), s[0], M[12]);
    M[13] = lz_fma2(Y, s[2], M[13]);
    M[14] = lz_fma2(Z, s[2], M[14]);
    M[15] = lz_fma2(Y2, s[1], M[15]);
    M[16] = lz_fma2(lz_dup(y2 * z), s[0], M[16]);
    M[17] = lz_fma2(Z2, s[1], M[17]);
    M[18] = lz_fma2(lz_dup(y * z2), s[0], M[18]);
    M[19] = lz_fma2(YZ, s[1], M[19]);
    const float2 Q = lz_dup(q);
    const float2 t2 = lz_fma2(Q, s[0], s[2]), t3 = lz_fma2(Q, s[1], s[3]);
    M[20] = lz_add2(M[20], lz_fma2(Q, s[2], s[4]));
    M[21] = lz_fma2(Y2, t2, M[21]);
    M[22] = lz_fma2(Z2, t2, M[22]);
    M[23] = lz_fma2(Y, t3, M[23]);
    M[24] = lz_fma2(Z, t3, M[24]);
    M[25] = lz_fma2(YZ, t2, M[25]);
}

// lz_warp_reduce_scatter for two cells at once.
__device__ __forceinline__ float2 lz_warp_reduce_scatter2(float2 (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float2 send = up ? v[i] : v[i + o];
            const float2 keep = up ? v[i + o] : v[i];
            v[i] = make_float2(keep.x + __shfl_xor_sync(0xFFFFFFFFu, send.x, o),
                               keep.y + __shfl_xor_sync(0xFFFFFFFFu, send.y, o));
        }
    }
    return v[0];
}

// Shared-memory accesses by 32-bit shared address.
__device__ __forceinline__ void lz_cp16s(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void lz_sts4(uint32_t dst, float v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "f"(v) : "memory");
}
__device__ __forceinline__ void lz_cp8s(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void lz_sts2(uint32_t dst, float v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %1};" ::"r"(dst), "f"(v) : "memory");
}
__device__ __forceinline__ float2 lz_lds2(uint32_t src)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(src) : "memory");
    return v;
}
// A thread's node vector: VW = 4 or 2 values.
template <int VW>
__device__ __forceinline__ void lz_cps(uint32_t dst, const void *src)
{
    if (VW == 4) lz_cp16s(dst, src);
    else lz_cp8s(dst, src);
}
template <int VW>
__device__ __forceinline__ void lz_stsv(uint32_t dst, float v)
{
    if (VW == 4) lz_sts4(dst, v);
    else lz_sts2(dst, v);
}
__device__ __forceinline__ float4 lz_lds4(uint32_t src)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(src)
                 : "memory");
    return v;
}

// A streaming thread's constant geometry.
struct LzQuad {
    int S, J, Jh, P4, pl, N, jy;
    bool yup, streams;
    int64_t pbytes;             // bytes per cell (N^3 floats)
    int sbytes;                 // bytes per stage of a cell (S node vectors)
    uint32_t ring0, ring_end;   // shared addresses: this thread's slots of ring slot 0; ring end
    uint32_t src;               // bytes between the three sources of a stage
    int stages;
};

// Prefetch position of a thread: cell pk of the group, stage pst of that
// cell, the shared address of the slots it fills next, and what the cell's
// sources are (cells, or a wall's ghost values).
struct LzPf {
    int pk, pst;
    int sidx;                // ring slot index of the next stage (bulk-copy ring)
    uint32_t slot;
    const char *own;         // this thread's quad of stage pst of cell pk
    int64_t xoff, yoff;      // byte offsets of the x and y source cells
    float gx, gxl;           // ghost values of the x source's wall, and of the left one (cells at a wall)
    const float *gy;         // ghost values of the bottom or top wall, by jx (cells at a wall)
    bool xin, xin_l, yin;    // the x source (and the left one) and the y source are cells
};

// v_x < 0 (the first half of the stages): the x source is the right cell;
// the half ends in lz_prefetch.
__device__ __forceinline__ void lz_pf_cell(LzPf &p, const LzQuad &q, const Geo &g, const LzArgs &a,
                                           const int4 *cells, const char *hin_t)
{
    const int4 ce = cells[p.pk];
    p.own = hin_t + (int64_t)ce.x * q.pbytes;
    p.xoff = q.pbytes;
    p.xin = ce.y < g.nx - 1;
    p.xin_l = ce.y > 0;
    p.yin = q.yup ? ce.z > 0 : ce.z < g.ny - 1;
    p.yoff = q.yup ? -(int64_t)g.nx * q.pbytes : (int64_t)g.nx * q.pbytes;
    p.gx = p.xin ? 0.f : __ldg(a.ghost + (g.ny + ce.z) * q.N + q.jy);
    p.gxl = p.xin_l ? 0.f : __ldg(a.ghost + ce.z * q.N + q.jy);
    p.gy = a.ghost + (q.yup ? 2 * g.ny + ce.y : 2 * g.ny + g.nx + ce.y) * q.N + q.pl;
}

// Stages this thread's own, x-source and y-source quads of the next stage
// (a wall's ghost value where the source lies outside the cavity) and
// commits one group of copies (an empty one past the group's last stage).
template <int VW>
__device__ __forceinline__ void lz_prefetch(LzPf &p, const LzQuad &q, const Geo &g, const LzArgs &a,
                                            const int4 *cells, const char *hin_t, int ncell)
{
    if (q.streams && p.pk < ncell) {
        if (p.pst == 0) lz_pf_cell(p, q, g, a, cells, hin_t);
        lz_cps<VW>(p.slot, p.own);
        if (p.xin) lz_cps<VW>(p.slot + q.src, p.own + p.xoff);
        else lz_stsv<VW>(p.slot + q.src, p.gx);
        if (p.yin) lz_cps<VW>(p.slot + 2 * q.src, p.own + p.yoff);
        else lz_stsv<VW>(p.slot + 2 * q.src, __ldg(p.gy + p.pst * q.P4));
        p.own += q.sbytes;
    }
    lz_cp_commit();
    p.slot += 3 * q.src;
    if (p.slot == q.ring_end) p.slot = q.ring0;
    ++p.pst;
    if (p.pst == q.Jh) {                         // v_x > 0 from here on: the left cell
        p.xoff = -q.pbytes;
        p.xin = p.xin_l;
        p.gx = p.gxl;
    }
    if (p.pst == q.J) {
        p.pst = 0;
        ++p.pk;
    }
}

// The producer's view of the bulk-copy ring: per slot (one bit each),
// whether a stage was issued into it whose reading has not been awaited yet,
// the parity of the next phase of its empty barrier, and the parity of its
// issue count.
struct LzTmaProd {
    uint32_t pending, epar, ipar;
};

// The same step with bulk copies: thread 0 of the role issues the stage's
// runs once every streaming warp has read the slot's previous stage.  The
// own and the x-source runs are S float4 each, contiguous in global memory
// and in the slot (a stage never straddles jx = N/2).  The y source differs
// within a plane: its rows jy < N/2 (v_y < 0) come from the cell above and
// its rows jy >= N/2 from the cell below, so each of the stage's P4 planes
// takes two half-plane copies.  Each thread still writes its wall ghost
// values into its own bytes of the slot (no copy where the source lies
// outside the cavity).
__device__ __forceinline__ void lz_prefetch_tma(LzPf &p, const LzQuad &q, const Geo &g, const LzArgs &a,
                                                const int4 *cells, const char *hin_t, int ncell, LzHead &H,
                                                LzTmaProd &pr)
{
    if (p.pk < ncell) {
        if (p.pst == 0) lz_pf_cell(p, q, g, a, cells, hin_t);
        const bool left = p.pst >= q.Jh, xin = p.xin;
        if (q.streams) {
            if (!xin) lz_sts4(p.slot + q.src, p.gx);
            if (!p.yin) lz_sts4(p.slot + 2 * q.src, __ldg(p.gy + p.pst * q.P4));
        }
        // After a wait gave up, nothing more is issued (the waits are skipped).
        if (threadIdx.x == 0 && *(volatile int *)&H.tma_err == 0) {
            const int s = p.sidx;
            const uint32_t full = lz_saddr(&H.bar_full[s]);
            if (pr.pending >> s & 1u) {
                lz_ring_wait(lz_saddr(&H.bar_empty[s]), pr.epar >> s & 1u, H.tma_err);
                pr.epar ^= 1u << s;
            }
            const uint32_t extra = (blockIdx.x == 0 && pr.ipar == 0u && pr.pending == 0u) ? (uint32_t)a.tx_excess : 0u;
            pr.pending |= 1u << s;
            pr.ipar ^= 1u << s;
            const uint32_t sb = (uint32_t)q.sbytes;
            const uint32_t hb = (uint32_t)(q.N * q.N) * 2u;          // half a plane (N^2/2 floats)
            const int4 ce = cells[p.pk];
            const bool above = ce.z < g.ny - 1, below = ce.z > 0;
            const uint32_t ybytes = (uint32_t)q.P4 * hb * ((above ? 1u : 0u) + (below ? 1u : 0u));
            lz_mbar_expect_tx(full, sb * (1u + (xin ? 1u : 0u)) + ybytes + extra);
            lz_bulk_g2s(p.slot, p.own, sb, full);
            if (xin) lz_bulk_g2s(p.slot + q.src, left ? p.own - q.pbytes : p.own + q.pbytes, sb, full);
            const int64_t ystep = (int64_t)g.nx * q.pbytes;
            for (int pl = 0; pl < q.P4; ++pl) {
                const uint32_t o = (uint32_t)pl * 2u * hb;
                if (above) lz_bulk_g2s(p.slot + 2 * q.src + o, p.own + ystep + o, hb, full);
                if (below) lz_bulk_g2s(p.slot + 2 * q.src + o + hb, p.own - ystep + o + hb, hb, full);
            }
        }
        p.own += q.sbytes;
    }
    p.slot += (3 * q.src);
    if (++p.sidx == q.stages) {
        p.sidx = 0;
        p.slot = q.ring0;
    }
    ++p.pst;
    if (p.pst == q.Jh) {
        p.xoff = -q.pbytes;
        p.xin = p.xin_l;
        p.gx = p.gxl;
    }
    if (p.pst == q.J) {
        p.pst = 0;
        ++p.pk;
    }
}

// Per-cell state of a thread's streaming: the (v_y, v_z) parts of the
// sources' pending corrections and the power sums over jx of N = w h~ /
// (A_y A_z) for the vector's node pairs.
template <int VW> struct LzAcc {
    float2 bdo[VW / 2], bdx[VW / 2], bdy[VW / 2];
    float2 s0[VW / 2], s1[VW / 2], s2[VW / 2], s3[VW / 2], s4[VW / 2];
};

// One streaming stage of one cell (Eq. streaming2D with the deferred
// correction applied to its sources): h~ to dst, the power sums, and the
// active nodes of the quad to the compact array (component k of G).  SX:
// stretched cells, the x Courant numbers times the cell's factor fx2.
template <int G, bool SX, int VW>
__device__ __forceinline__ void lz_stream_stage(uint32_t sl, uint32_t src, int jx, int j0, int k, const LzHead &H,
                                                const float4 *tcx, const float2 *tcy, LzAcc<VW> &c,
                                                char *dst, const uint2 *smask, float *Af,
                                                float2 eps2, float2 one2, float2 nay2, float2 fx2)
{
    float2 h0p[VW / 2], hxp[VW / 2], hyp[VW / 2];
    if constexpr (VW == 4) {
        const float4 h0 = lz_lds4(sl), hx = lz_lds4(sl + src), hy = lz_lds4(sl + 2 * src);
        h0p[0] = lz_lo(h0); h0p[1] = lz_hi(h0);
        hxp[0] = lz_lo(hx); hxp[1] = lz_hi(hx);
        hyp[0] = lz_lo(hy); hyp[1] = lz_hi(hy);
    } else {
        h0p[0] = lz_lds2(sl);
        hxp[0] = lz_lds2(sl + src);
        hyp[0] = lz_lds2(sl + 2 * src);
    }
    const float4 cx4 = tcx[jx];
    const float2 cy2 = tcy[jx];
    const float4 ta = H.ta[jx];
    const float2 nax2 = SX ? lz_mul2(lz_lo(ta), fx2) : lz_lo(ta), A2 = lz_hi(ta);
    const float4 v12 = H.tv12[jx], v34 = H.tv34[jx];
    float2 ht[VW / 2];
    const float2 mone2 = lz_dup(-1.f);
#pragma unroll
    for (int p = 0; p < VW / 2; ++p) {
        // u = h_c + (1 + eps h_c) kappa of each source, as h_c (1 + eps kappa) + kappa.
        const float2 ko = lz_add2(lz_lo(cx4), c.bdo[p]);
        const float2 u0 = lz_fma2(h0p[p], lz_fma2(eps2, ko, one2), ko);
        const float2 kx = lz_add2(lz_hi(cx4), c.bdx[p]);
        const float2 ux = lz_fma2(hxp[p], lz_fma2(eps2, kx, one2), kx);
        const float2 ky = lz_add2(cy2, c.bdy[p]);
        const float2 uy = lz_fma2(hyp[p], lz_fma2(eps2, ky, one2), ky);
        // Eq. streaming2D: u0 - ax (u0 - ux) - ay (u0 - uy).
        float2 h = lz_fma2(nax2, lz_fma2(ux, mone2, u0), u0);
        h = lz_fma2(nay2, lz_fma2(uy, mone2, u0), h);
        ht[p] = h;
        const float2 n = lz_mul2(h, A2);
        c.s0[p] = lz_add2(c.s0[p], n);
        c.s1[p] = lz_fma2(n, lz_lo(v12), c.s1[p]);
        c.s2[p] = lz_fma2(n, lz_hi(v12), c.s2[p]);
        c.s3[p] = lz_fma2(n, lz_lo(v34), c.s3[p]);
        c.s4[p] = lz_fma2(n, lz_hi(v34), c.s4[p]);
    }
    if constexpr (VW == 4) *reinterpret_cast<float4 *>(dst) = make_float4(ht[0].x, ht[0].y, ht[1].x, ht[1].y);
    else *reinterpret_cast<float2 *>(dst) = ht[0];
    // Active nodes of the quad (nodes j0 .. j0 + 3) go to the compact array.
    const uint2 mw = smask[j0 >> 5];
    const int sh = j0 & 31;
    const uint32_t bits = (mw.x >> sh) & ((1u << VW) - 1u);
    if (bits) {
        int mi = (int)mw.y + __popc(mw.x & ((1u << sh) - 1u));
#pragma unroll
        for (int i = 0; i < VW; ++i)
            if (bits >> i & 1u) Af[(mi++) * G + k] = i & 1 ? ht[i / 2].y : ht[i / 2].x;
    }
}

// g = ha + hb + eps ha hb per cell, as ha + hb (1 + eps ha), and acc += w g
// (Eq. monteCarloInt: the sample's product, signed and weighted for its
// destination).
__device__ __forceinline__ void lz_term(float2 ha, float2 hb, float2 eps2, float2 w2, float2 &acc)
{
    const float2 g = lz_fma2(hb, lz_fma2(eps2, ha, lz_dup(1.f)), ha);
    acc = lz_fma2(w2, g, acc);
}
__device__ __forceinline__ void lz_term(float4 ha, float4 hb, float2 eps2, float2 w2, float4 &acc)
{
    float2 lo = lz_lo(acc), hi = lz_hi(acc);
    lz_term(lz_lo(ha), lz_lo(hb), eps2, w2, lo);
    lz_term(lz_hi(ha), lz_hi(hb), eps2, w2, hi);
    acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The state of a thread's run: the sum of its current destination and the
// shared addresses where that and the next destination's go.  A destination
// ends with one predicated store.  (With an atomic branch for the first
// destination in each of the 24 unrolled terms, the terms of four cells took
// 104 thousand cycles at 32^3 and 2x10^4 samples instead of 61.)  Neighbouring
// runs may share a thread's first destination and its unfinished last one, so
// the first sum goes to a slot of the thread's own (at first p is the slot);
// both are added to the increments atomically at the end of the run.
template <typename V> struct LzRun {
    V acc;
    uint32_t p, next;
};
__device__ __forceinline__ void lz_sts(uint32_t dst, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void lz_sts(uint32_t dst, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(v.x), "f"(v.y) : "memory");
}

template <typename V>
__device__ __forceinline__ void lz_apply(V ha, V hb, uint2 r, float2 eps2, LzRun<V> &st)
{
    lz_term(ha, hb, eps2, lz_dup(__uint_as_float(r.y)), st.acc);
    if (r.x & 1u) {                              // the destination's last term
        lz_sts(st.p, st.acc);
        st.p = st.next;
        st.next += sizeof(V);
        lz_set_zero(st.acc);
    }
}

// Applies 8 records (the operands of two terms are read before either of
// them can store a destination's sum).
template <typename V, uint32_t AMASK>
__device__ __forceinline__ void lz_apply8(const uint2 (&r)[8], const char *Ab, float2 eps2, LzRun<V> &st)
{
#pragma unroll
    for (int h = 0; h < 8; h += 2) {
        const V ha0 = *reinterpret_cast<const V *>(Ab + (r[h].x & AMASK));
        const V hb0 = *reinterpret_cast<const V *>(Ab + (r[h].x >> 16));
        const V ha1 = *reinterpret_cast<const V *>(Ab + (r[h + 1].x & AMASK));
        const V hb1 = *reinterpret_cast<const V *>(Ab + (r[h + 1].x >> 16));
        lz_apply(ha0, hb0, r[h], eps2, st);
        lz_apply(ha1, hb1, r[h + 1], eps2, st);
    }
}

// Barriers among the threads of one role (named barrier 1: streaming, 2:
// collision; 0 is __syncthreads).
template <int ST>
__device__ __forceinline__ void lz_stream_bar() { asm volatile("bar.sync 1, %0;" ::"n"(ST) : "memory"); }
__device__ __forceinline__ void lz_coll_bar() { asm volatile("bar.sync 2, %0;" ::"n"(kLzCollT) : "memory"); }
// Named barrier 3 over all threads: the collision role arrives without
// waiting once its terms are complete; the streaming role waits for that.
template <int ST>
__device__ __forceinline__ void lz_terms_done_arrive()
{
    asm volatile("bar.arrive 3, %0;" ::"n"(lz_threads(ST)) : "memory");
}
template <int ST>
__device__ __forceinline__ void lz_terms_done_wait()
{
    asm volatile("bar.sync 3, %0;" ::"n"(lz_threads(ST)) : "memory");
}
constexpr int kLzTailChunk = 256;  // active nodes per claimed chunk of the increment sums

// One CTA per SM, two roles working on consecutive groups of G cells: the first
// ST / 32 warps stream group i (Eq. streaming2D, the power sums, the active nodes
// to one compact array), while the last eight solve the correction and the
// moments of group i - 2 (a warp per cell) and then apply the collision terms,
// their sums and the write-back of group i - 1 from the other compact array.
// Streaming is bound by HBM and its instructions and the collision terms by
// shared memory, so the two overlap.
//
// NV: the velocity axis length as a compile-time constant (0: read g.nv at
// run time).  SX: stretched cells (per-column and per-row Courant factors
// g.sx, g.sy).  Streaming thread t < S = K N^2/4 owns node quad q = t mod
// (N^2/4) (four consecutive jz at one (jx, jy)) of jx-plane t div (N^2/4) of
// every stage; a stage covers K planes and a cell J = N / K stages.  VW = 2: node
// pairs in place of quads, N^2/2 of them to a plane.
//
// TMA: the streaming sources arrive by bulk copies (cp.async.bulk) that
// thread 0 of the role issues into a ring of slots, with a full
// and an empty mbarrier per slot, instead of per-thread cp.async.
//
// lz_run runs the pipeline of one CTA over the groups grp0, grp0 + gstride,
// ... (nmine of them) of one problem; the kernel k_lz gives CTA b the groups
// b, b + gridDim.x, ...
template <int G, int NV, bool SX, int ST, bool TMA = false, int VW = NV % 4 == 0 ? 4 : 2>
__device__ __forceinline__ void lz_run(const Geo &g, const LzArgs &a, char *smem_raw, int grp0, int gstride,
                                       int nmine)
{
    using V = typename LzVec<G>::T;
    constexpr int kThreads = lz_threads(ST), kStreamWarps = ST / 32;
    if (a.meta[1]) {                              // too many active nodes: k_cell4 runs
        if (a.fb_count)
            for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < a.fb_n; i += gridDim.x * blockDim.x)
                a.fb_count[i] = 0;
        return;
    }
    const int N = NV ? NV : g.nv;
    const int N2 = N * N, nvt = N2 * N, t = threadIdx.x;
    const int Qd = N2 / VW, nq = N / VW, P4 = lz_planes(N, ST), J = N / P4, Jh = J / 2;
    const int S = P4 * Qd;                        // node vectors per stage (the threads that stream)
    const int half = N / 2;
    LzHead &H = *reinterpret_cast<LzHead *>(smem_raw);
    const int M = a.meta[0];
    const LzOff so = lz_offsets(nvt, a.mcap, G, a.stages, S, VW);
    V *Bv = reinterpret_cast<V *>(smem_raw + so.bc);
    float *Bf = reinterpret_cast<float *>(smem_raw + so.bc);
    uint2 *smask = reinterpret_cast<uint2 *>(smem_raw + so.mask);   // mask word, compact index of its first node
    uint16_t *sact = reinterpret_cast<uint16_t *>(smem_raw + so.act);
    const float eps = g.epsf;
    const float2 eps2 = lz_dup(eps), one2 = lz_dup(1.f);
    const int lane = t & 31, warp = t >> 5;
    const bool streamer = t < ST;

    // ---- tables (once per launch) ----------------------------------------
    for (int i = t; i < N; i += kThreads) {
        const double v = g.axv[i], A = g.axA[i];
        // Courant numbers 0 without streaming: h~ is then exactly the
        // corrected input (every source term is multiplied by zero).
        const float nax = a.nostream ? 0.f : -(float)fabs(v * g.dt / g.dx), fA = (float)A, fv = (float)v;
        H.v[i] = fv;
        H.A[i] = fA;
        H.IA[i] = (float)(1.0 / A);
        H.cuy[i] = a.nostream ? 0.f : (float)fabs(v * g.dt / (SX ? g.dx : g.dy));
        H.ta[i] = make_float4(nax, nax, fA, fA);
        const float v2 = (float)(v * v), v3 = (float)(v * v * v), v4 = (float)(v * v * v * v);
        H.tv12[i] = make_float4(fv, fv, v2, v2);
        H.tv34[i] = make_float4(v3, v3, v4, v4);
    }
    for (int w = t; w < (nvt + 31) / 32; w += kThreads) {
        smask[w] = make_uint2(a.mask[w], (uint32_t)a.wpre[w]);
    }
    for (int m = t; m < M; m += kThreads) {     // active nodes as jx << 10 | jy << 5 | jz
        const int j = a.act[m], jxy = j / N, jx = jxy / N;
        sact[m] = (uint16_t)(jx << 10 | (jxy - jx * N) << 5 | (j - jxy * N));
    }
    for (int i = t; i < 2 * kLzMaxG * kLzDParts * 32; i += kThreads) (&H.dpart[0][0][0][0])[i] = 0.f;
    if (t < kLzX) H.e0[t] = a.e0[t];
    if (t < 50) H.px[t / 10][t % 10] = (unsigned char)lz_psiphi(t / 10, t % 10);
    if (TMA && t == 0) {
        for (int s = 0; s < a.stages; ++s) {
            lz_mbar_init(lz_saddr(&H.bar_full[s]), 1);
            lz_mbar_init(lz_saddr(&H.bar_empty[s]), kStreamWarps);
        }
        H.tma_err = 0;
        lz_mbar_init_fence();
    }
    __syncthreads();

    // A streaming thread's quad.
    const bool streams = t < S;
    const int pl = streams ? t / Qd : 0, q = streams ? t - pl * Qd : 0;
    const int jy = q / nq, jz = VW * (q - jy * nq);
    const bool yup = jy >= half;                  // v_y > 0: the y source is below
    const float2 nay2 = lz_dup(-H.cuy[jy]);
    int fallback = 0;
    LzTmaProd prod{0u, 0u, 0u};                   // thread 0: the bulk-copy ring's producer state
    uint32_t fpar = 0u;                           // parity of each slot's next full phase

    // One warp per cell of group it - 2: totals over the warps, then the
    // correction and the moments (k: the warp's number within its role).
    auto solve = [&](int it, int k) {
        if (it < 2) return;
        const int grp = grp0 + (it - 2) * gstride, fb = (it - 2) % 3, db = it & 1, kc = grp * G + k;
        if (k >= G || kc >= g.nr) return;
        if (lane < kLzMono) {
            // Compensated totals over the warps: T = F + D (the sums of N_c)
            // and D.
            const float f = H.ftot[fb][k][0][lane], fc = H.ftot[fb][k][1][lane];
            float d = 0.f, dc = 0.f;
#pragma unroll
            for (int w = 0; w < kLzDParts; ++w) {
                float e;
                two_sum(d, H.dpart[db][k][w][lane], d, e);
                dc = __fadd_rn(dc, e);
            }
            float tt, te, hi, lo;
            two_sum(f, d, tt, te);
            two_sum(tt, __fadd_rn(te, __fadd_rn(fc, dc)), hi, lo);
            H.ftot[fb][k][0][lane] = hi;
            H.ftot[fb][k][1][lane] = lo;
            H.dpart[db][k][0][lane] = __fadd_rn(d, dc);
        }
        __syncwarp();
        lz_finish(g, a, cell_of(g, kc), H.ftot[fb][k][0], H.ftot[fb][k][1], H.dpart[db][k][0], H.e0, &H.px[0][0],
                  &fallback);
        __syncwarp();
        // The slots take the increment sums of a later group (atomically).
        for (int i = lane; i < kLzDParts * 32; i += 32) (&H.dpart[db][k][0][0])[i] = 0.f;
    };

    // Iteration it: the streaming warps take this CTA's group it, the
    // collision warps its group it - 1.
    for (int it = 0; it <= nmine + 1; ++it) {
        const bool clk = a.clk && grp0 == 0 && it < kClkCells;
        if (clk && t == 0) a.clk[it * kClkPhases + 0] = clock64();
        if (streamer) {
            if (it < nmine) {
                const int grp = grp0 + it * gstride, buf = it & 1;
                float *Af = reinterpret_cast<float *>(smem_raw + kLzAOff + buf * so.abytes);
                if (t < G) {
                    const int kc = grp * G + t;
                    const int c = kc < g.nr ? cell_of(g, kc) : -1;
                    H.cell[buf][t] = make_int4(c, c >= 0 ? c % g.nx : 0, c >= 0 ? c / g.nx : 0, 0);
                }
                lz_stream_bar<ST>();
                int ncell = 0;
#pragma unroll
                for (int k = 0; k < G; ++k) ncell += H.cell[buf][k].x >= 0 ? 1 : 0;
                // mu of the five cells each cell's streaming reads (0 outside the cavity).
                for (int i = t; i < G * 40; i += ST) {
                    const int k = i / 40, r = i - k * 40, s5 = r / 8, m = r - s5 * 8;
                    const int4 ce = H.cell[buf][k];
                    int cs = ce.x;
                    bool ok = ce.x >= 0 && m < 5;
                    if (s5 == 1) { ok = ok && ce.y < g.nx - 1; cs = ce.x + 1; }
                    if (s5 == 2) { ok = ok && ce.y > 0; cs = ce.x - 1; }
                    if (s5 == 3) { ok = ok && ce.z > 0; cs = ce.x - g.nx; }
                    if (s5 == 4) { ok = ok && ce.z < g.ny - 1; cs = ce.x + g.nx; }
                    H.mus[k][s5][m] = ok ? a.mu_in[(int64_t)cs * 8 + m] : 0.f;
                }
                // a.stages - 1 stages in flight ahead of the one being used.
                const uint32_t ring0 = lz_saddr(smem_raw + so.ring) + t * (VW * 4);
                const LzQuad qd{S, J, Jh, P4, pl, N, jy, yup, streams, (int64_t)nvt * 4, S * VW * 4, ring0,
                                ring0 + a.stages * 3 * S * VW * 4, (uint32_t)(S * VW * 4), a.stages};
                const char *hin_t = reinterpret_cast<const char *>(a.hin) + t * (VW * 4);
                LzPf pf{};
                pf.slot = ring0;
                const int4 *cells = H.cell[buf];
#pragma unroll 1
                for (int kk = 0; kk < a.stages - 1; ++kk) {
                    if (TMA) lz_prefetch_tma(pf, qd, g, a, cells, hin_t, ncell, H, prod);
                    else lz_prefetch<VW>(pf, qd, g, a, cells, hin_t, ncell);
                }
                lz_stream_bar<ST>();
                // Correction tables of the group's cells: ca(jx) = mu_0 + mu_x
                // v_x + mu_4 v_x^2 of the own cell, the upwind x cell (right for
                // jx < N/2, left otherwise), and the cells below and above.
                for (int i = t; i < G * N; i += ST) {
                    const int k = i / N, jx = i - k * N;
                    const float vx = H.v[jx];
                    float ca[5];
#pragma unroll
                    for (int s5 = 0; s5 < 5; ++s5) {
                        const float *m = H.mus[k][s5];
                        ca[s5] = m[0] + m[1] * vx + m[4] * vx * vx;
                    }
                    const float cx = jx < half ? ca[1] : ca[2];
                    H.tcx[k][jx] = make_float4(ca[0], ca[0], cx, cx);
                    H.tcy[k][0][jx] = lz_dup(ca[3]);
                    H.tcy[k][1][jx] = lz_dup(ca[4]);
                }
                lz_stream_bar<ST>();

                // ---- streaming with the deferred correction applied to its sources
                uint32_t cslot = ring0;           // slots of the stage being used
                int cidx = 0;                     // and their index
#pragma unroll 1
                for (int k = 0; k < ncell; ++k) {
                    // A cell at a wall had ghost values written into its slots
                    // by the threads (generic proxy) before later bulk copies.
                    const int4 cek = cells[k];
                    const bool wallk = TMA && (cek.y == 0 || cek.y == g.nx - 1 || cek.z == 0 || cek.z == g.ny - 1);
                    LzAcc<VW> ac;
#pragma unroll
                    for (int p = 0; p < VW / 2; ++p)
                        ac.s0[p] = ac.s1[p] = ac.s2[p] = ac.s3[p] = ac.s4[p] = lz_zero2();
                    lz_bd<VW>(H.mus[k][0], H.v, jy, jz, ac.bdo);
                    lz_bd<VW>(H.mus[k][1], H.v, jy, jz, ac.bdx);
                    lz_bd<VW>(H.mus[k][yup ? 3 : 4], H.v, jy, jz, ac.bdy);
                    const float4 *tcx = H.tcx[k];
                    const float2 *tcy = H.tcy[k][yup ? 0 : 1];
                    char *dst = reinterpret_cast<char *>(a.hout) + (int64_t)cells[k].x * nvt * 4 + t * (VW * 4);
                    // Courant factors of this cell on stretched grids.
                    float2 fx2 = one2, nay2k = nay2;
                    if (SX) {
                        fx2 = lz_dup((float)g.sx[cells[k].y]);
                        nay2k = lz_dup(-H.cuy[jy] * (float)g.sy[cells[k].z]);
                    }
                    int jx = pl, j0 = VW * t;
#pragma unroll 1
                    for (int st = 0; st < J; ++st) {
                        if (st == Jh) lz_bd<VW>(H.mus[k][2], H.v, jy, jz, ac.bdx);   // the left cell now
                        // The slots read last stage take the stage a.stages - 1
                        // ahead; then this stage's copies have landed.
                        if (TMA) {
                            lz_prefetch_tma(pf, qd, g, a, cells, hin_t, ncell, H, prod);
                            lz_ring_wait(lz_saddr(&H.bar_full[cidx]), fpar >> cidx & 1u, H.tma_err);
                            fpar ^= 1u << cidx;
                        } else {
                            lz_prefetch<VW>(pf, qd, g, a, cells, hin_t, ncell);
                            lz_cp_wait_but(a.stages - 1);
                        }
                        if (streams)
                            lz_stream_stage<G, SX, VW>(cslot, qd.src, jx, j0, k, H, tcx, tcy, ac, dst, smask, Af,
                                                   eps2, one2, nay2k, fx2);
                        if (TMA) {
                            // The warp has read the slot: release it to the producer.
                            if (wallk) lz_fence_proxy_async();
                            __syncwarp();
                            if (lane == 0) lz_mbar_arrive(lz_saddr(&H.bar_empty[cidx]));
                        }
                        cslot += 3 * qd.src;
                        if (TMA) {
                            if (++cidx == a.stages) {
                                cidx = 0;
                                cslot = ring0;
                            }
                        } else if (cslot == qd.ring_end) {
                            cslot = ring0;
                        }
                        jx += P4;
                        j0 += VW * S;
                        dst += S * VW * 4;
                    }
                    // The 26 monomial sums of the thread's nodes, summed over the warp.
                    float Msum[32];
#pragma unroll
                    for (int r = 0; r < 32; ++r) Msum[r] = 0.f;
                    if (streams) {
                        const float Ay = H.A[jy];
#pragma unroll
                        for (int i = 0; i < VW; ++i) {
                            const int p = i / 2;
                            const float Ayz = Ay * H.A[jz + i];
                            const float sv[5] = {i & 1 ? ac.s0[p].y : ac.s0[p].x, i & 1 ? ac.s1[p].y : ac.s1[p].x,
                                                 i & 1 ? ac.s2[p].y : ac.s2[p].x, i & 1 ? ac.s3[p].y : ac.s3[p].x,
                                                 i & 1 ? ac.s4[p].y : ac.s4[p].x};
                            float si[5];
#pragma unroll
                            for (int pp = 0; pp < 5; ++pp) si[pp] = sv[pp] * Ayz;
                            lz_mono_from_powers(si, H.v[jy], H.v[jz + i], Msum);
                        }
                    }
                    H.fpart[k][warp][lane] = lz_warp_reduce_scatter(Msum);
                }
                if (!TMA) lz_cp_wait_all();
                // Compensated totals over the warps, one warp per cell.
                lz_stream_bar<ST>();
                if (warp < G && lane < kLzMono) {
                    float f = 0.f, fc = 0.f;
#pragma unroll
                    for (int w = 0; w < kStreamWarps; ++w) {
                        float e;
                        two_sum(f, H.fpart[warp][w][lane], f, e);
                        fc = __fadd_rn(fc, e);
                    }
                    H.ftot[it % 3][warp][0][lane] = f;
                    H.ftot[it % 3][warp][1][lane] = fc;
                }
            }
            if (clk && t == 0) a.clk[it * kClkPhases + 1] = clock64();
        } else {
            solve(it, warp - kStreamWarps);
            if (clk && t == ST) a.clk[it * kClkPhases + 5] = clock64();
        }
        if (!streamer && it >= 1 && it <= nmine) {
            const int tc = t - ST, buf = (it - 1) & 1;
            char *Ab = smem_raw + kLzAOff + buf * so.abytes;
            float *Af = reinterpret_cast<float *>(Ab);
            int ncell = 0, cg[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                cg[k] = H.cell[buf][k].x;
                ncell += cg[k] >= 0 ? 1 : 0;
            }
            // ---- Monte Carlo terms (Eq. monteCarloInt) ----------------------
            // The increments start from zero; the zero entry M of h~ stands for
            // nodes outside the grid, and cells missing from a short group hold 0.
            for (int i = tc; i < M + 1; i += kLzCollT) lz_set_zero(Bv[i]);
            if (tc < G) Af[M * G + tc] = 0.f;
            if (tc == 0) H.tail_next = 0;
            if (ncell < G)
                for (int i = tc; i < M * G; i += kLzCollT)
                    if (i % G >= ncell) Af[i] = 0.f;
            lz_coll_bar();
            {
                // Each thread applies its run of the destination-sorted terms:
                // it sums one destination's terms in registers and stores the
                // sum when the destination's last term has passed (LzRun).
                const int C = a.meta[3];
                if (C > 0) {
                    constexpr uint32_t amask = G == 4 ? 0xFFF0u : 0xFFF8u;
                    LzRun<V> st;
                    // The slot: 16 bytes of the increment sums' slots, idle
                    // (zero) until the terms are done.
                    V *const first = reinterpret_cast<V *>(&H.dpart[buf][0][0][0] + 4 * tc);
                    const int dest0 = a.dest0[tc];
                    const uint32_t slot = lz_saddr(first);
                    lz_set_zero(st.acc);
                    st.p = slot;
                    st.next = lz_saddr(Bv + dest0 + 1);
                    // Batches of 8 records in three register buffers: a buffer
                    // is refilled as soon as it has been applied, two batches
                    // ahead (the records stream from L2).  A run is C records,
                    // C a multiple of 8, zero-padded by the plan.
                    const uint2 *rp = a.rec + tc;
                    constexpr int Ts = kLzCollT, Bs = 8 * kLzCollT;
                    uint2 r0[8], r1[8], r2[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        r0[u] = rp[u * Ts];
                        r1[u] = C > 8 ? rp[Bs + u * Ts] : make_uint2(0u, 0u);
                        r2[u] = C > 16 ? rp[2 * Bs + u * Ts] : make_uint2(0u, 0u);
                    }
                    for (int i = 0; i < C; i += 24) {
                        rp += 3 * Bs;
                        lz_apply8<V, amask>(r0, Ab, eps2, st);
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (i + 24 < C) r0[u] = rp[u * Ts];
                        if (i + 8 < C) {
                            lz_apply8<V, amask>(r1, Ab, eps2, st);
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (i + 32 < C) r1[u] = rp[Bs + u * Ts];
                        }
                        if (i + 16 < C) {
                            lz_apply8<V, amask>(r2, Ab, eps2, st);
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (i + 40 < C) r2[u] = rp[2 * Bs + u * Ts];
                        }
                    }
                    const bool ended = st.p != slot;      // the first destination's sum is in the slot
                    lz_atomic_add(ended ? Bv + (st.p - lz_saddr(Bv)) / sizeof(V) : Bv + dest0, st.acc);
                    if (ended) {
                        lz_atomic_add(Bv + dest0, *first);
                        lz_set_zero(*first);
                    }
                }
            }
            if (clk && tc == 0) a.clk[it * kClkPhases + 2] = clock64();
            if (a.early_tail) {
                // The increments are complete once every collision thread is here.
                lz_coll_bar();
                lz_terms_done_arrive<ST>();
            }
        }
        // ---- sums of the collision increment and h_c = h~ + dN / w on the
        // active nodes of group it - 1, two cells at a time.  Either all
        // warps after a CTA barrier, each with a fixed share of the nodes and
        // its partial sums added to the slots of warp (warp mod 8); or
        // (early tail, the default: the collision terms take less time than the
        // streaming) the collision warps as soon as their terms are complete and the streaming warps once they are
        // done, every warp claiming chunks of kLzTailChunk nodes of one cell
        // pair at a time (pair 0 first) and adding its partial sums of a pair
        // to the slots when it moves on.
        if (it >= 1 && it <= nmine) {
            const bool early = a.early_tail;
            if (early) {
                if (streamer) lz_terms_done_wait<ST>();
            } else {
                __syncthreads();
            }
            const int buf = (it - 1) & 1;
            const float *Af = reinterpret_cast<const float *>(smem_raw + kLzAOff + buf * so.abytes);
            int ncell = 0, cg[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                cg[k] = H.cell[buf][k].x;
                ncell += cg[k] >= 0 ? 1 : 0;
            }
            if (!early) {
                const int u = streamer ? t + kLzCollT : t - ST;
#pragma unroll
                for (int k2 = 0; k2 < G; k2 += 2) {
                    float2 D2[32];
#pragma unroll
                    for (int r = 0; r < 32; ++r) D2[r] = lz_zero2();
                    if (k2 < ncell) {
                        for (int mm = u; mm < M; mm += kThreads) {
                            const int pk = sact[mm], jx = pk >> 10, jyy = pk >> 5 & 31, jz = pk & 31;
                            const int j = (jx * N + jyy) * N + jz;
                            const float2 d = *reinterpret_cast<const float2 *>(Bf + mm * G + k2);
                            const float2 h = *reinterpret_cast<const float2 *>(Af + mm * G + k2);
                            const float x = H.v[jx], x2 = x * x;
                            const float2 sp[5] = {d, lz_mul2(d, lz_dup(x)), lz_mul2(d, lz_dup(x2)),
                                                  lz_mul2(d, lz_dup(x2 * x)), lz_mul2(d, lz_dup(x2 * x2))};
                            lz_mono_from_powers2(sp, H.v[jyy], H.v[jz], D2);
                            const float iw = H.IA[jx] * H.IA[jyy] * H.IA[jz];
                            a.hout[(int64_t)cg[k2] * nvt + j] = fmaf(d.x, iw, h.x);
                            if (k2 + 1 < ncell) a.hout[(int64_t)cg[k2 + 1] * nvt + j] = fmaf(d.y, iw, h.y);
                        }
                    }
                    const float2 r = lz_warp_reduce_scatter2(D2);
                    atomicAdd(&H.dpart[buf][k2][warp & (kLzDParts - 1)][lane], r.x);
                    atomicAdd(&H.dpart[buf][k2 + 1][warp & (kLzDParts - 1)][lane], r.y);
                }
            } else {
                const int npair = (ncell + 1) / 2, per = (M + kLzTailChunk - 1) / kLzTailChunk;
                const int nchunk = npair * per;
                float2 D2[32];
#pragma unroll
                for (int r = 0; r < 32; ++r) D2[r] = lz_zero2();
                int kcur = -1;
                for (;;) {
                    int ch = 0;
                    if (lane == 0) ch = atomicAdd(&H.tail_next, 1);
                    ch = __shfl_sync(0xFFFFFFFFu, ch, 0);
                    const int k2 = ch < nchunk ? 2 * (ch / per) : -1;
                    if (k2 != kcur) {
                        if (kcur >= 0) {
                            const float2 r = lz_warp_reduce_scatter2(D2);
                            atomicAdd(&H.dpart[buf][kcur][warp & (kLzDParts - 1)][lane], r.x);
                            atomicAdd(&H.dpart[buf][kcur + 1][warp & (kLzDParts - 1)][lane], r.y);
#pragma unroll
                            for (int r2 = 0; r2 < 32; ++r2) D2[r2] = lz_zero2();
                        }
                        kcur = k2;
                    }
                    if (k2 < 0) break;
                    const int m0 = (ch - (k2 / 2) * per) * kLzTailChunk, m1 = min(M, m0 + kLzTailChunk);
                    for (int mm = m0 + lane; mm < m1; mm += 32) {
                        const int pk = sact[mm], jx = pk >> 10, jyy = pk >> 5 & 31, jz = pk & 31;
                        const int j = (jx * N + jyy) * N + jz;
                        const float2 d = *reinterpret_cast<const float2 *>(Bf + mm * G + k2);
                        const float2 h = *reinterpret_cast<const float2 *>(Af + mm * G + k2);
                        const float x = H.v[jx], x2 = x * x;
                        const float2 sp[5] = {d, lz_mul2(d, lz_dup(x)), lz_mul2(d, lz_dup(x2)),
                                              lz_mul2(d, lz_dup(x2 * x)), lz_mul2(d, lz_dup(x2 * x2))};
                        lz_mono_from_powers2(sp, H.v[jyy], H.v[jz], D2);
                        const float iw = H.IA[jx] * H.IA[jyy] * H.IA[jz];
                        a.hout[(int64_t)cg[k2] * nvt + j] = fmaf(d.x, iw, h.x);
                        if (k2 + 1 < ncell) a.hout[(int64_t)cg[k2 + 1] * nvt + j] = fmaf(d.y, iw, h.y);
                    }
                }
            }
            if (clk && t == ST) a.clk[it * kClkPhases + 3] = clock64();
            if (clk && t == ST) a.clk[it * kClkPhases + 4] = clock64();
        }
        __syncthreads();
    }
    if (fallback && a.stats) atomicAdd(a.stats + 3, (unsigned long long)fallback);
    if (TMA && t == 0 && H.tma_err) {
        // A wait gave up: report it, and wait (bounded) for the last copy
        // issued into each slot before the CTA leaves (after the first
        // timeout nothing more was issued).
        if (a.err) atomicOr(a.err, 1ull);
        for (int s = 0; s < a.stages; ++s)
            if (prod.pending >> s & 1u) lz_mbar_wait(lz_saddr(&H.bar_full[s]), (prod.ipar >> s & 1u) ^ 1u);
    }
}

template <int G, int NV, bool SX, int ST, bool TMA = false, int VW = NV % 4 == 0 ? 4 : 2>
__global__ void __launch_bounds__(lz_threads(ST), 1) k_lz(const __grid_constant__ Geo g, const __grid_constant__ LzArgs a)
{
    extern __shared__ __align__(16) char smem_raw[];
    const int ngroups = (g.nr + G - 1) / G;
    const int nmine = blockIdx.x < ngroups ? (ngroups - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    lz_run<G, NV, SX, ST, TMA, VW>(g, a, smem_raw, blockIdx.x, gridDim.x, nmine);
}

}  // namespace bzk
