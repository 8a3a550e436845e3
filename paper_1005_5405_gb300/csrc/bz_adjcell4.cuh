// bz_adjcell4.cuh -- one step's adjoint, FP32 states with a velocity axis that is
// a multiple of 4 (Eqs. streaming2D, monteCarloInt, collision_step, rinorm_a,
// correzione and their transposes).
//
// k_adj_cell4 takes a cell from lam = dJ/dh^{n+1} to dJ/dh~ in three slabs of
// shared memory, A (h~, read by every phase), B and C:
//   stream h^n                  A = h~, C = 0
//   g_l W_l of every sample     B
//   forward terms by node       C = dN (sum of +-g_l W_l)
//   one pass over the nodes     B = lam; sums of N_c = w h~ + dN (14), of dN (5)
//                               and of nu = lam (1 + eps h_c) psi (5), in one reduction
//   two solves of G             mu = -G^-1 D and xi = G^-1 nu, a warp each
//   lam_c / w                   B = q
//   gamma_l of every sample     C
//   loss terms by node          B = sum of gamma_l (1 + eps h~_p)
//   one pass over the nodes     dJ/dh~ = lam_c + w psi.xi + B
// with, in the cell (lam_j, psi = 1, v, v^2; h_c = h~ + dN / w):
//   lam_c,j = (lam_j - w_j psi_j.xi)(1 + eps psi_j.mu),  q = lam_c / w
//   dJ/dh~_j = lam_c,j + w_j psi_j.xi
//   gamma_l = W_l (q_a* + q_b* - q_a - q_b)
//   dJ/dh~_a += gamma_l (1 + eps h~_b),  dJ/dh~_b += gamma_l (1 + eps h~_a).
// A thread owns quads of four jz nodes of one jy row in J consecutive jx-planes
// (quads of a row are rotated by jx so that gathers spread over the banks).
//
// Bound: latency between ten barriers and the shared-memory gathers (17.0
// thousand wavefronts of a cell's 30 thousand cycles at 20^3 with 5000 samples,
// two CTAs of 512 threads an SM); HBM needs only 0.5 of its 1.8 ms a step at
// 128^2.  Against the forward kernel's body with a transposed tail (gathers twice
// per loss term, three reductions, two solves by one lane after another, sums
// flushed by branches): four steps of 128^2 x 20^3 8.66 -> 7.24 ms.  A w (q + psi.xi)
// pass in place of reading lam twice was as fast, but w times 1 / w is off by the
// same rounding in every step: 5 times the error over 8 steps.
#pragma once

#include "bz_lazy.cuh"

namespace bzk {

// The step's lists, in node positions of the rotated slab order.  Per sample
// (in place of the plan's records): lossW = {4a | 4b << 16, W} and gain = {4a* |
// 4b* << 16, -}, byte offsets, 4 nvt (a zero) for a node outside the grid.  The
// forward terms, sorted by node: node << 18 | loss << 17 | l << 2; the loss terms,
// sorted by node d in {a, b}: {d << 18 | l << 2, byte offset of the other node}.
// 14 bits of node and 15 of sample: nvt < 16384 (three slabs of a larger grid do
// not fit shared memory), nt <= 32768.  Thread t of the cell kernel reads its
// contiguous run of C entries in groups of 16 bytes (4 forward, 2 loss terms) at a
// stride of T groups.  Counts, cursors and headers {E, C} of
// the loss list come nvt entries (two ints) after those of the forward list.
static __global__ void k_adj_count2(int nt, int nvt, const ushort4 *__restrict__ pidx,
                                    int *__restrict__ count)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nt) return;
    const ushort4 q = pidx[l];
    if (q.x != 0xFFFF) {
        atomicAdd(count + q.x, 1);
        atomicAdd(count + nvt + q.x, 1);
    }
    if (q.y != 0xFFFF) {
        atomicAdd(count + q.y, 1);
        atomicAdd(count + nvt + q.y, 1);
    }
    if (q.z != 0xFFFF) atomicAdd(count + q.z, 1);
    if (q.w != 0xFFFF) atomicAdd(count + q.w, 1);
}
static __global__ void __launch_bounds__(1024) k_adj_scan2(int nvt, int T, const int *__restrict__ count,
                                                           int *__restrict__ cursor, int *__restrict__ meta)
{
    __shared__ int part[1024];
    const int k = blockIdx.x;
    scatter_scan_body(nvt, T, count + k * nvt, cursor + k * nvt, meta + 2 * k, part);
}
static __global__ void k_adj_fill2(int nt, int nvt, int T, ushort4 *__restrict__ pidx,
                                   PlanA<float, uint16_t> *__restrict__ pa, int *__restrict__ cursor,
                                   const int *__restrict__ meta, uint32_t *__restrict__ ent,
                                   uint2 *__restrict__ rec)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nt) return;
    const ushort4 q = pidx[l];
    const unsigned short d[4] = {q.x, q.y, q.z, q.w};
    const int C = meta[1], CL = meta[3];
    auto off = [&](unsigned short i) { return 4u * (i != 0xFFFF ? (uint32_t)i : (uint32_t)nvt); };
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (d[k] == 0xFFFF) continue;
        const int pos = atomicAdd(cursor + d[k], 1), tt = pos / C, i = pos - tt * C;
        ent[((int64_t)(i >> 2) * T + tt) * 4 + (i & 3)] = ((uint32_t)d[k] << 18) | (k < 2 ? 0x20000u : 0u) | ((uint32_t)l << 2);
        if (k < 2) {
            const int pl = atomicAdd(cursor + nvt + d[k], 1), tl = pl / CL, il = pl - tl * CL;
            rec[((int64_t)(il >> 1) * T + tl) * 2 + (il & 1)] = make_uint2(((uint32_t)d[k] << 18) | ((uint32_t)l << 2), off(d[1 - k]));
        }
    }
    const float W = pa[l].W;
    reinterpret_cast<uint2 *>(pidx)[l] = make_uint2(off(q.x) | off(q.y) << 16, __float_as_uint(W));
    reinterpret_cast<uint2 *>(pa)[l] = make_uint2(off(q.z) | off(q.w) << 16, 0u);
}

struct Adj4Smem {
    float4 *A, *B, *C;   // slabs of nvt (+ 4: zeros after A and B)
    float *gw0, *gw1;    // products of the forward terms, gamma (in B and C when nt <= nvt)
    float *slot;         // kMaxThreads: a run's first sum; partial sums of the reduction
    float *tot;          // 32 sums
    float *sol;          // mu [8], xi [8]
    float *G0;           // 25: the Gram matrix of the equilibrium
    float4 *pw;          // N: {v, v^2, v^3, v^4}
    float2 *aia;         // N: {A, 1/A}
    float2 *ca;          // N: {mu_x v + mu_4 v^2, xi_x v + xi_4 v^2} of the cell
    float *v, *Az, *IAz, *cu;   // N each
    int4 *cell;          // the cell (index, ix, iy), found by one thread
};
__host__ __device__ inline size_t adj4_smem(Adj4Smem *s, char *base, int N, int nvt, int nt)
{
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 15) & ~(size_t)15; return base + o; };
    Adj4Smem x;
    x.A = (float4 *)take(4 * (size_t)(nvt + 4));
    x.B = (float4 *)take(4 * (size_t)(nvt + 4));
    x.C = (float4 *)take(4 * (size_t)nvt);
    const bool in = nt <= nvt;
    x.gw0 = in ? (float *)x.B : (float *)take(4 * (size_t)nt);
    x.gw1 = in ? (float *)x.C : x.gw0;
    x.slot = (float *)take(4 * kMaxThreads);
    x.tot = (float *)take(128);
    x.sol = (float *)take(64);
    x.G0 = (float *)take(100);
    x.pw = (float4 *)take(16 * N);
    x.aia = (float2 *)take(8 * N);
    x.ca = (float2 *)take(8 * N);
    x.v = (float *)take(4 * N);
    x.Az = (float *)take(4 * N);
    x.IAz = (float *)take(4 * N);
    x.cu = (float *)take(4 * N);
    x.cell = (int4 *)take(16);
    if (s) *s = x;
    return off;
}
__host__ __device__ inline size_t adj4_smem_bytes(int nv, int nvt, int nt)
{
    return adj4_smem(nullptr, nullptr, nv, nvt, nt);
}

// The pivoted solves of mu and xi (solve 0 and 8 entries in), by one thread.
static __device__ __noinline__ void adj4_solve_fallback(const Geo *g, const float *tot, float *sol, int *fallback)
{
    double P[19], x[5];
    int f2 = 0;
    for (int k = 0; k < 19; ++k) P[k] = (double)tot[k];
    correction_solve<float>(*g, P, x, &f2);
    for (int k = 0; k < 5; ++k) sol[k] = (float)x[k];
    f2 = 0;
    for (int k = 0; k < 5; ++k) P[14 + k] = -(double)tot[19 + k];
    correction_solve<float>(*g, P, x, &f2);
    for (int k = 0; k < 5; ++k) sol[8 + k] = (float)x[k];
    *fallback += 1 + f2;
}

// mu = -G^-1 D and xi = G^-1 nu from the 24 sums (tot[24]: room for one more), by a
// warp: Gauss-Jordan elimination without pivoting (G is symmetric positive
// definite) with a column a lane: 0-4 those of G, 5 and 6 the right-hand sides,
// 7-11 the identity; then one step of refinement with residuals evaluated exactly
// and rounded once (as correction_spd), row a on lane a (mu) and 16 + a (xi).  The
// chain is 5 broadcasts and reciprocals: a solve by every lane took 11 thousand of
// a cell's 66 thousand cycles.
__device__ __forceinline__ void adj4_solve(const Geo &g, const Adj4Smem &S, int *fallback)
{
    const unsigned all = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    float *tot = S.tot, *sol = S.sol;
    if (lane == 0) tot[24] = tot[4] + tot[5] + tot[6];
    __syncwarp();
    const int j = lane & 15;
    auto pack = [](uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e) {
        return a | b << 5 | c << 10 | d << 15 | e << 20;
    };
    uint32_t mi = pack(0, 1, 2, 3, 24);              // sums of column j of G
    mi = j == 1 ? pack(1, 4, 7, 8, 10) : mi;
    mi = j == 2 ? pack(2, 7, 5, 9, 11) : mi;
    mi = j == 3 ? pack(3, 8, 9, 6, 12) : mi;
    mi = j == 4 ? pack(24, 10, 11, 12, 13) : mi;
    float a[5], u[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a[i] = j < 5 ? S.G0[j * 5 + i] + g.epsf * tot[mi >> (5 * i) & 31u] : 0.f;
        u[i] = a[i];
        if (lane == 5) u[i] = -tot[14 + i];
        if (lane == 6) u[i] = tot[19 + i];
        if (lane == 7 + i) u[i] = 1.f;
    }
    const float b = j < 5 ? (lane < 16 ? -tot[14 + j] : tot[19 + j]) : 0.f;
    bool ok = g.solve_fb == 0;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const float piv = __shfl_sync(all, u[k], k);
        ok = ok && piv > 0.f;
        u[k] *= 1.f / piv;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            if (i == k) continue;
            const float f = __shfl_sync(all, u[i], k);
            u[i] = fmaf(-f, u[k], u[i]);
        }
    }
    if (!ok) {
        if (lane == 0) adj4_solve_fallback(&g, tot, sol, fallback);
        __syncwarp();
        return;
    }
    float hi = b, lo = 0.f;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const float x = __shfl_sync(all, u[c], lane < 16 ? 5 : 6);
        float p, pe, s, se;
        two_prod(a[c], x, p, pe);
        two_sum(hi, -p, s, se);
        hi = s;
        lo = __fadd_rn(lo, __fsub_rn(se, pe));
    }
    const float r = __fadd_rn(hi, lo);
    float dm = 0.f, dx = 0.f;
#pragma unroll
    for (int c = 0; c < 5; ++c) {                    // (row a of the inverse: its column a)
        dm = fmaf(u[c], __shfl_sync(all, r, c), dm);
        dx = fmaf(u[c], __shfl_sync(all, r, 16 + c), dx);
    }
    if (lane == 5 || lane == 6) {
#pragma unroll
        for (int c = 0; c < 5; ++c) sol[(lane - 5) * 8 + c] = u[c];
    }
    __syncwarp();
    if (lane >= 7 && lane < 12) {
        sol[lane - 7] += dm;
        sol[lane + 1] += dx;
    }
    __syncwarp();
}

__device__ __forceinline__ float adj4_hsum(float2 a) { return a.x + a.y; }
__device__ __forceinline__ float2 adj4_sub2(float2 a, float2 b) { return lz_fma2(b, lz_dup(-1.f), a); }

// A thread's run of n terms, in groups of 16 bytes at stride T, summed by node
// into base.  A finished node is one predicated store; neighbouring runs may share
// the first and the last node, so the first sum goes to the thread's slot and both
// are added atomically at the end.  Two groups are in flight while the previous two
// are summed.
__device__ __forceinline__ void adj4_step(uint32_t w, float r, uint32_t base, uint32_t &prev, uint32_t &p, float &acc)
{
    asm volatile("{\n .reg .pred q;\n .reg .b32 x;\n xor.b32 x, %3, %2;\n setp.ge.u32 q, x, 0x40000;\n"
                 " @q st.shared.f32 [%0], %1;\n shr.u32 x, %3, 16;\n and.b32 x, x, 0xFFFC;\n"
                 " @q add.u32 %0, x, %5;\n @q mov.f32 %1, 0f00000000;\n add.rn.f32 %1, %1, %4;\n}"
                 : "+r"(p), "+f"(acc) : "r"(prev), "r"(w), "f"(r), "r"(base) : "memory");
    prev = w;
}
__device__ __forceinline__ uint32_t adj4_key(uint4 e, int u, uint32_t)
{
    return u == 0 ? e.x : u == 1 ? e.y : u == 2 ? e.z : e.w;
}
__device__ __forceinline__ uint2 adj4_key(uint4 e, int u, uint2)
{
    return u == 0 ? make_uint2(e.x, e.y) : make_uint2(e.z, e.w);
}
__device__ __forceinline__ uint32_t adj4_word(uint32_t e) { return e; }
__device__ __forceinline__ uint32_t adj4_word(uint2 e) { return e.x; }
template <typename E, typename VAL>
__device__ __forceinline__ void adj4_run(int n, const uint4 *__restrict__ list, int T, float *basef, float *slot, VAL val)
{
    constexpr int PG = 16 / sizeof(E), CH = 2 * PG;
    if (n <= 0) return;
    const uint32_t base = lz_saddr(basef), sl = lz_saddr(slot);
    const int last = (n - 1) / PG;
    uint4 e[2], f[2];
    e[0] = list[0];
    e[1] = list[(int64_t)min(1, last) * T];
    const uint32_t first = adj4_word(adj4_key(e[0], 0, E{}));
    uint32_t prev = first, p = sl;
    float acc = 0.f;
    for (int i = 0; i < n; i += CH) {
#pragma unroll
        for (int u = 0; u < 2; ++u) f[u] = list[(int64_t)min(i / PG + 2 + u, last) * T];
        if (i + CH <= n) {
            float r[CH];
#pragma unroll
            for (int u = 0; u < CH; ++u) r[u] = val(adj4_key(e[u / PG], u % PG, E{}));
#pragma unroll
            for (int u = 0; u < CH; ++u) adj4_step(adj4_word(adj4_key(e[u / PG], u % PG, E{})), r[u], base, prev, p, acc);
        } else {
#pragma unroll
            for (int u = 0; u < CH; ++u)
                if (i + u < n) {
                    const E x = adj4_key(e[u / PG], u % PG, E{});
                    adj4_step(adj4_word(x), val(x), base, prev, p, acc);
                }
        }
        e[0] = f[0];
        e[1] = f[1];
    }
    atomicAdd(basef + (prev >> 18), acc);
    if (p != sl) atomicAdd(basef + (first >> 18), *slot);
}

template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1024 / MAXT)
k_adj_cell4(const __grid_constant__ Geo g, Map4 m, const float *__restrict__ hin,
            const float *__restrict__ ghost, const uint2 *__restrict__ lossW,
            const uint2 *__restrict__ gain, const uint4 *__restrict__ ent,
            const int *__restrict__ meta, const uint4 *__restrict__ lrec,
            const float *__restrict__ lam, float *__restrict__ lt,
            unsigned long long *__restrict__ stats)
{
    extern __shared__ __align__(16) char smem_raw[];
    Adj4Smem S;
    adj4_smem(&S, smem_raw, g.nv, g.nvt, g.nt);
    const int N = g.nv, nvt = g.nvt, nt = g.nt, T = blockDim.x, t = threadIdx.x;
    for (int i = t; i < N; i += T) {
        const double v = g.axv[i], A = g.axA[i];
        S.pw[i] = make_float4((float)v, (float)(v * v), (float)(v * v * v), (float)(v * v * v * v));
        S.aia[i] = make_float2((float)A, (float)(1.0 / A));
        S.v[i] = (float)v;
        S.Az[i] = (float)A;
        S.IAz[i] = (float)(1.0 / A);
        S.cu[i] = (float)(v * g.dt / g.dx);
    }
    for (int i = t; i < 25; i += T) S.G0[i] = g.G0f[i];
    if (t < 4) reinterpret_cast<float *>(S.A)[nvt + t] = reinterpret_cast<float *>(S.B)[nvt + t] = 0.f;
    auto find = [&](int kc) {
        const int c = cell_of(g, kc), iy = c / g.nx;
        S.cell[0] = make_int4(c, c - iy * g.nx, iy, 0);
    };
    if (t == 0) find(blockIdx.x);
    __syncthreads();

    const int Q = m.Q, nq = N / 4, half = N / 2;
    const int kchunk = t / Q, q = t - kchunk * Q, jy = q / nq, qz = q - jy * nq;
    const bool active = kchunk < m.K;
    const int jx0 = active ? kchunk * m.J : 0, jx1 = active ? jx0 + m.J : 0;
    // Slab position of the quad in plane jx: jx Q + jy nq + (qz + jx) mod nq.
    const int r0 = (qz + jx0) % nq, row = jy * nq;
    const float eps = g.epsf;
    const float2 eps2 = lz_dup(eps);
    const int E = meta[0], C = meta[1], EL = meta[2], CL = meta[3];
    const int n = min(C, E - t * C), nl = min(CL, EL - t * CL);
    const int64_t plane = nvt / 4;
    int fallback = 0;

    for (int kc = blockIdx.x; kc < g.nr; kc += gridDim.x) {
        const int c = S.cell[0].x, ix = S.cell[0].y, iy = S.cell[0].z;
        // lam of the cell is needed two barriers later.
        for (int i = 32 * t; i < nvt; i += 32 * T)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(lam + (int64_t)c * nvt + i));

        const float4 *lam4 = reinterpret_cast<const float4 *>(lam) + (int64_t)c * plane;

        // ---- A = h~ (streaming), C = 0
        if (active) {
            const float4 *own = reinterpret_cast<const float4 *>(hin) + (int64_t)c * plane;
            const float fx = g.sx ? (float)g.sx[ix] : 1.f, fy = g.sy ? (float)g.sy[iy] : g.ryf;
            const float cuy = S.cu[jy] * fy, ay = fabsf(cuy);
            const bool xr = ix < g.nx - 1, xl = ix > 0, yi = cuy > 0.f ? iy > 0 : iy < g.ny - 1;
            const float4 *ys = own + (cuy > 0.f ? -(int64_t)g.nx : (int64_t)g.nx) * plane;
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            int r = r0;
            if (xr && xl && yi) {
#pragma unroll 4
                for (int jx = jx0; jx < jx1; ++jx) {
                    const int o = jx * Q + q, p = jx * Q + row + r;
                    const float4 h0 = own[o], hx = jx < half ? own[o + plane] : own[o - plane], hy = ys[o];
                    S.A[p] = upwind4(h0, hx, hy, fabsf(S.cu[jx]) * fx, ay);
                    S.C[p] = z4;
                    r = r + 1 == nq ? 0 : r + 1;
                }
            } else {
                const float *yg = ghost + (2 * g.ny + (cuy > 0.f ? 0 : g.nx) + ix) * N;
                for (int jx = jx0; jx < jx1; ++jx) {
                    const int o = jx * Q + q, p = jx * Q + row + r;
                    const float4 h0 = own[o], hy = yi ? ys[o] : f4(yg[jx]);
                    float4 hx;
                    if (jx < half) hx = xr ? own[o + plane] : f4(ghost[(g.ny + iy) * N + jy]);
                    else hx = xl ? own[o - plane] : f4(ghost[iy * N + jy]);
                    S.A[p] = upwind4(h0, hx, hy, fabsf(S.cu[jx]) * fx, ay);
                    S.C[p] = z4;
                    r = r + 1 == nq ? 0 : r + 1;
                }
            }
        }
        __syncthreads();

        // ---- g_l W_l on h~
        const char *Ab = reinterpret_cast<const char *>(S.A);
        for (int l0 = t; l0 < nt; l0 += 8 * T) {
            uint2 w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = l0 + u * T < nt ? lossW[l0 + u * T] : make_uint2(0u, 0u);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float ha = *reinterpret_cast<const float *>(Ab + (w[u].x & 0xFFFFu));
                const float hb = *reinterpret_cast<const float *>(Ab + (w[u].x >> 16));
                if (l0 + u * T < nt) S.gw0[l0 + u * T] = fmaf(hb, fmaf(eps, ha, 1.f), ha) * __uint_as_float(w[u].y);
            }
        }
        __syncthreads();

        // ---- C = dN, the forward terms summed by node
        {
            const char *gb = reinterpret_cast<const char *>(S.gw0);
            adj4_run<uint32_t>(n, ent + t, T, reinterpret_cast<float *>(S.C), S.slot + t, [&](uint32_t w) {
                const uint32_t r = *reinterpret_cast<const uint32_t *>(gb + (w & 0x1FFFCu));
                return __uint_as_float(r ^ (w << 14 & 0x80000000u));
            });
        }
        __syncthreads();

        // ---- B = lam; sums of lam (1 + eps h_c), then of N_c and dN (apart: the
        // sums of both and the tables do not fit 64 registers)
        const float vy = S.v[jy];
        {
            float M[32];
            const float4 zv = reinterpret_cast<const float4 *>(S.v)[qz];
            const float2 z0 = lz_lo(zv), z1 = lz_hi(zv), zz0 = lz_mul2(z0, z0), zz1 = lz_mul2(z1, z1);
            const float2 ayi = S.aia[jy];
            const float y2 = vy * vy;
            float e0 = 0.f, e1 = 0.f, ez = 0.f, e4 = 0.f;
            if (active) {
                const float4 iz = reinterpret_cast<const float4 *>(S.IAz)[qz];
                const float2 i0 = lz_mul2(lz_dup(ayi.y), lz_lo(iz)), i1 = lz_mul2(lz_dup(ayi.y), lz_hi(iz));
                int r = r0;
#pragma unroll 4
                for (int jx = jx0; jx < jx1; ++jx) {
                    const int p = jx * Q + row + r;
                    r = r + 1 == nq ? 0 : r + 1;
                    const float4 l = lam4[jx * Q + q], h = S.A[p], d = S.C[p];
                    S.B[p] = l;
                    const float4 x = S.pw[jx];
                    const float2 ix2 = lz_dup(S.aia[jx].y), L0 = lz_lo(l), L1 = lz_hi(l);
                    const float2 g0 = lz_fma2(lz_mul2(ix2, i0), lz_lo(d), lz_lo(h));   // h_c
                    const float2 g1 = lz_fma2(lz_mul2(ix2, i1), lz_hi(d), lz_hi(h));
                    const float2 t0 = lz_fma2(lz_mul2(L0, eps2), g0, L0), t1 = lz_fma2(lz_mul2(L1, eps2), g1, L1);
                    const float u = adj4_hsum(lz_add2(t0, t1));
                    e0 += u;
                    e1 = fmaf(u, x.x, e1);
                    e4 = fmaf(u, x.y, e4) + adj4_hsum(lz_fma2(t0, zz0, lz_mul2(t1, zz1)));
                    ez += adj4_hsum(lz_fma2(t0, z0, lz_mul2(t1, z1)));
                }
            }
            M[19] = e0;
            M[20] = e1;
            M[21] = vy * e0;
            M[22] = ez;
            M[23] = fmaf(y2, e0, e4);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, a4 = 0.f, b0 = 0.f, b1 = 0.f, b2 = 0.f;
            float c0 = 0.f, c1 = 0.f, c2 = 0.f, s3 = 0.f, s4 = 0.f;
            float d0 = 0.f, d1 = 0.f, dz = 0.f, d4 = 0.f;
            if (active) {
                const float4 az = reinterpret_cast<const float4 *>(S.Az)[qz];
                const float2 w0 = lz_mul2(lz_dup(ayi.x), lz_lo(az)), w1 = lz_mul2(lz_dup(ayi.x), lz_hi(az));
                int r = r0;
#pragma unroll 1
                for (int jx = jx0; jx < jx1; ++jx) {
                    const int p = jx * Q + row + r;
                    r = r + 1 == nq ? 0 : r + 1;
                    const float4 h = S.A[p], d = S.C[p], x = S.pw[jx];
                    const float2 ax = lz_dup(S.aia[jx].x), D0 = lz_lo(d), D1 = lz_hi(d);
                    const float2 n0 = lz_fma2(lz_mul2(ax, w0), lz_lo(h), D0);
                    const float2 n1 = lz_fma2(lz_mul2(ax, w1), lz_hi(h), D1);
                    const float2 m0 = lz_mul2(n0, zz0), m1 = lz_mul2(n1, zz1);
                    const float s0 = adj4_hsum(lz_add2(n0, n1));
                    const float s1 = adj4_hsum(lz_fma2(n0, z0, lz_mul2(n1, z1)));
                    const float s2 = adj4_hsum(lz_add2(m0, m1));
                    a0 += s0;
                    a1 = fmaf(s0, x.x, a1);
                    a2 = fmaf(s0, x.y, a2);
                    a3 = fmaf(s0, x.z, a3);
                    a4 = fmaf(s0, x.w, a4);
                    b0 += s1;
                    b1 = fmaf(s1, x.x, b1);
                    b2 = fmaf(s1, x.y, b2);
                    c0 += s2;
                    c1 = fmaf(s2, x.x, c1);
                    c2 = fmaf(s2, x.y, c2);
                    s3 += adj4_hsum(lz_fma2(m0, z0, lz_mul2(m1, z1)));
                    s4 += adj4_hsum(lz_fma2(m0, zz0, lz_mul2(m1, zz1)));
                    const float u = adj4_hsum(lz_add2(D0, D1));
                    d0 += u;
                    d1 = fmaf(u, x.x, d1);
                    d4 = fmaf(u, x.y, d4) + adj4_hsum(lz_fma2(D0, zz0, lz_mul2(D1, zz1)));
                    dz += adj4_hsum(lz_fma2(D0, z0, lz_mul2(D1, z1)));
                }
            }
            const float q0 = fmaf(y2, a0, c0), q1 = fmaf(y2, a1, c1), q2 = fmaf(y2, a2, c2);
            M[0] = a0;
            M[1] = a1;
            M[2] = vy * a0;
            M[3] = b0;
            M[4] = a2;
            M[5] = y2 * a0;
            M[6] = c0;
            M[7] = vy * a1;
            M[8] = b1;
            M[9] = vy * b0;
            M[10] = a3 + q1;
            M[11] = vy * (a2 + q0);
            M[12] = b2 + fmaf(y2, b0, s3);
            M[13] = a4 + 2.f * q2 + fmaf(y2, fmaf(y2, a0, 2.f * c0), s4);
            M[14] = d0;
            M[15] = d1;
            M[16] = vy * d0;
            M[17] = dz;
            M[18] = fmaf(y2, d0, d4);
#pragma unroll
            for (int k = 24; k < 32; ++k) M[k] = 0.f;
            S.slot[t] = lz_warp_reduce_scatter(M);
        }
        __syncthreads();

        // ---- mu and xi, and their tables (first warp)
        if (t < 32) {
            float f = 0.f, fc = 0.f;                 // compensated sum of the warps' sums
#pragma unroll 8
            for (int w = 0; w < T / 32; ++w) {
                float e;
                two_sum(f, S.slot[w * 32 + t], f, e);
                fc = __fadd_rn(fc, e);
            }
            S.tot[t] = __fadd_rn(f, fc);
            __syncwarp();
            adj4_solve(g, S, &fallback);
            for (int i = t; i < N; i += 32) {
                const float4 x = S.pw[i];
                S.ca[i] = make_float2(S.sol[1] * x.x + S.sol[4] * x.y, S.sol[9] * x.x + S.sol[12] * x.y);
            }
            if (t == 0 && kc + gridDim.x < g.nr) find(kc + gridDim.x);
        }
        __syncthreads();

        // ---- B = q = lam_c / w
        // (px, pm: psi.xi and psi.mu without the part of v_x, which is in S.ca)
        const float2 one = lz_dup(1.f);
        float2 px0, px1, pm0, pm1;
        {
            const float4 zv = reinterpret_cast<const float4 *>(S.v)[qz];
            auto part = [&](const float *s, float2 z) {
                const float2 k = lz_dup(s[0] + s[2] * vy + s[4] * vy * vy);
                return lz_fma2(lz_fma2(lz_dup(s[4]), z, lz_dup(s[3])), z, k);
            };
            px0 = part(S.sol + 8, lz_lo(zv));
            px1 = part(S.sol + 8, lz_hi(zv));
            pm0 = part(S.sol, lz_lo(zv));
            pm1 = part(S.sol, lz_hi(zv));
        }
        if (active) {
            const float4 iz = reinterpret_cast<const float4 *>(S.IAz)[qz];
            const float2 ayi = S.aia[jy];
            const float2 i0 = lz_mul2(lz_dup(ayi.y), lz_lo(iz)), i1 = lz_mul2(lz_dup(ayi.y), lz_hi(iz));
            int r = r0;
#pragma unroll 2
            for (int jx = jx0; jx < jx1; ++jx) {
                const int p = jx * Q + row + r;
                r = r + 1 == nq ? 0 : r + 1;
                const float4 l = S.B[p];
                const float2 cc = S.ca[jx], iax = lz_dup(S.aia[jx].y);
                const float2 m0 = lz_fma2(eps2, lz_add2(pm0, lz_dup(cc.x)), one);
                const float2 m1 = lz_fma2(eps2, lz_add2(pm1, lz_dup(cc.x)), one);
                const float2 x0 = lz_add2(px0, lz_dup(cc.y)), x1 = lz_add2(px1, lz_dup(cc.y));
                // (lam / w - psi.xi) (1 + eps psi.mu)
                const float2 v0 = lz_mul2(lz_fma2(lz_mul2(iax, i0), lz_lo(l), make_float2(-x0.x, -x0.y)), m0);
                const float2 v1 = lz_mul2(lz_fma2(lz_mul2(iax, i1), lz_hi(l), make_float2(-x1.x, -x1.y)), m1);
                S.B[p] = make_float4(v0.x, v0.y, v1.x, v1.y);
            }
        }
        __syncthreads();

        // ---- gamma_l
        {
            const char *Bb = reinterpret_cast<const char *>(S.B);
            auto at = [&](uint32_t o) { return *reinterpret_cast<const float *>(Bb + o); };
            for (int l0 = t; l0 < nt; l0 += 5 * T) {
                uint2 w[5];
                uint32_t v[5];
#pragma unroll
                for (int u = 0; u < 5; ++u) {
                    const int l = l0 + u * T < nt ? l0 + u * T : l0;
                    w[u] = lossW[l];
                    v[u] = gain[l].x;
                }
#pragma unroll
                for (int u = 0; u < 5; ++u) {
                    const float s = (at(v[u] & 0xFFFFu) + at(v[u] >> 16)) - (at(w[u].x & 0xFFFFu) + at(w[u].x >> 16));
                    if (l0 + u * T < nt) S.gw1[l0 + u * T] = __uint_as_float(w[u].y) * s;
                }
            }
        }
        __syncthreads();

        // ---- B = 0 for the loss terms
        if (active) {
            int r = r0;
            for (int jx = jx0; jx < jx1; ++jx) {
                S.B[jx * Q + row + r] = make_float4(0.f, 0.f, 0.f, 0.f);
                r = r + 1 == nq ? 0 : r + 1;
            }
        }
        // The next cell's own state will be read by streaming first.
        if (kc + gridDim.x < g.nr) {
            for (int i = 32 * t; i < nvt; i += 32 * T)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(hin + (int64_t)S.cell[0].x * nvt + i));
        }
        __syncthreads();

        // ---- B = the loss terms summed by node
        {
            const char *gb = reinterpret_cast<const char *>(S.gw1);
            adj4_run<uint2>(nl, lrec + t, T, reinterpret_cast<float *>(S.B), S.slot + t, [&](uint2 w) {
                const float gam = *reinterpret_cast<const float *>(gb + (w.x & 0x1FFFCu));
                const float hp = *reinterpret_cast<const float *>(Ab + w.y);
                return gam * fmaf(eps, hp, 1.f);
            });
        }
        __syncthreads();

        // ---- dJ/dh~ = lam_c + w psi.xi + B.  (From lam again: w (lam_c / w) would
        // carry the rounding of w times 1 / w, the same in every step.)
        if (active) {
            float4 *dst = reinterpret_cast<float4 *>(lt) + (int64_t)c * plane;
            const float4 az = reinterpret_cast<const float4 *>(S.Az)[qz];
            const float ay = S.aia[jy].x;
            const float2 w0 = lz_mul2(lz_dup(ay), lz_lo(az)), w1 = lz_mul2(lz_dup(ay), lz_hi(az));
            int r = r0;
#pragma unroll 4
            for (int jx = jx0; jx < jx1; ++jx) {
                const int o = jx * Q + q;
                const float4 l = lam4[o], b = S.B[jx * Q + row + r];
                r = r + 1 == nq ? 0 : r + 1;
                const float2 cc = S.ca[jx], ax = lz_dup(S.aia[jx].x);
                const float2 m0 = lz_fma2(eps2, lz_add2(pm0, lz_dup(cc.x)), one);
                const float2 m1 = lz_fma2(eps2, lz_add2(pm1, lz_dup(cc.x)), one);
                const float2 y0 = lz_mul2(lz_mul2(ax, w0), lz_add2(px0, lz_dup(cc.y)));
                const float2 y1 = lz_mul2(lz_mul2(ax, w1), lz_add2(px1, lz_dup(cc.y)));
                const float2 v0 = lz_add2(lz_fma2(adj4_sub2(lz_lo(l), y0), m0, y0), lz_lo(b));
                const float2 v1 = lz_add2(lz_fma2(adj4_sub2(lz_hi(l), y1), m1, y1), lz_hi(b));
                dst[o] = make_float4(v0.x, v0.y, v1.x, v1.y);
            }
        }
    }
    if (fallback && stats) atomicAdd(stats + 3, (unsigned long long)fallback);
}

// dJ/dh^n from dJ/dh~ (FP32, velocity axis a multiple of 4): the transposed
// upwind stencil (h^n_c feeds h~ of its downwind neighbours: right for v_x >
// 0, above for v_y > 0) in 16-byte quads of four jz nodes, plus on boundary
// cells the outgoing-flux terms lF[f] |v_n| w of their faces and on the lid
// row the lid-shear term wD 2 w v_x v_y / nx.  blockDim a multiple of Q.
static __global__ void __launch_bounds__(1024) k_adj_stream4(Geo g, const float *__restrict__ lt,
                                                             const double *__restrict__ lF,
                                                             float *__restrict__ lam_out, double wD)
{
    __shared__ float sv[kMaxN], sax[kMaxN], say[kMaxN], sA[kMaxN];
    const int N = g.nv, nq = N / 4, Q = N * N / 4, half = N / 2;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const double v = g.axv[i];
        sv[i] = (float)v;
        sax[i] = (float)(fabs(v) * g.dt / g.dx);
        say[i] = (float)(fabs(v) * g.dt / g.dy);
        sA[i] = (float)g.axA[i];
    }
    __syncthreads();
    const int64_t plane = g.nvt / 4;
    const int q = threadIdx.x % Q, jxs = threadIdx.x / Q, jstep = blockDim.x / Q;
    const int jy = q / nq, jz0 = 4 * (q % nq);
    const float vy = sv[jy], ay = say[jy];
    const float dcoef = (float)(wD * 2.0 / g.nx);
    for (int kc = blockIdx.x; kc < g.nr; kc += gridDim.x) {
        const int c = cell_of(g, kc);
        const int ix = c % g.nx, iy = c / g.nx;
        const float4 *own = reinterpret_cast<const float4 *>(lt) + (int64_t)c * plane;
        float4 *dst = reinterpret_cast<float4 *>(lam_out) + (int64_t)c * plane;
        // Downwind y neighbour of this thread's row (v_y > 0: above).
        const float4 *ys = own + (jy >= half ? (int64_t)g.nx : -(int64_t)g.nx) * plane;
        if (ix > 0 && ix < g.nx - 1 && iy > 0 && iy < g.ny - 1) {
            // Interior cell: both downwind neighbours are cells.
            const float4 *xr = own + plane, *xl = own - plane;
#pragma unroll 4
            for (int jx = jxs; jx < N; jx += jstep) {
                const int o = jx * Q + q;
                const float ax = sax[jx];
                const float4 l0 = own[o], lx = jx >= half ? xr[o] : xl[o], ly = ys[o];
                const float c0 = 1.f - ax - ay;
                dst[o] = make_float4(c0 * l0.x + ax * lx.x + ay * ly.x, c0 * l0.y + ax * lx.y + ay * ly.y,
                                     c0 * l0.z + ax * lx.z + ay * ly.z, c0 * l0.w + ax * lx.w + ay * ly.w);
            }
            continue;
        }
        const bool yd = jy >= half ? iy < g.ny - 1 : iy > 0;
        for (int jx = jxs; jx < N; jx += jstep) {
            const int o = jx * Q + q;
            const float ax = sax[jx];
            const bool xd = jx >= half ? ix < g.nx - 1 : ix > 0;   // v_x > 0: right
            const float4 l0 = own[o];
            const float4 lx = xd ? own[o + (jx >= half ? plane : -plane)] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 ly = yd ? ys[o] : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 r;
            const float c0 = 1.f - ax - ay;
            r.x = c0 * l0.x + ax * lx.x + ay * ly.x;
            r.y = c0 * l0.y + ax * lx.y + ay * ly.y;
            r.z = c0 * l0.z + ax * lx.z + ay * ly.z;
            r.w = c0 * l0.w + ax * lx.w + ay * ly.w;
            const float vx = sv[jx];
            float ex = 0.f;
            if (ix == 0 && vx < 0.f) ex -= (float)lF[iy] * vx;
            if (ix == g.nx - 1 && vx > 0.f) ex += (float)lF[g.ny + iy] * vx;
            if (iy == 0 && vy < 0.f) ex -= (float)lF[2 * g.ny + ix] * vy;
            float dl = 0.f;
            if (iy == g.ny - 1 && vy > 0.f) {
                ex += (float)lF[2 * g.ny + g.nx + ix] * vy;
                dl = dcoef * vx * vy;
            }
            const float wxy = sA[jx] * sA[jy];
            float *rr = &r.x;
#pragma unroll
            for (int i = 0; i < 4; ++i) rr[i] += (ex + dl) * wxy * sA[jz0 + i];
            dst[o] = r;
        }
    }
}

}  // namespace bzk
