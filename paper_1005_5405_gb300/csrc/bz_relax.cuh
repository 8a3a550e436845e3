// bz_relax.cuh -- one step of a cell with the collision increments apart.
//
// Same mathematics as k_cell (Eqs. streaming2D, monteCarloInt,
// collision_step, rinorm_a, correzione, densita..sforzi) for the handles that
// the active-node kernel does not take: FP64 states, odd velocity axes and
// per-cell sample sets.  k_cell turns its slab into N = w h~, adds every
// sample's product to it with four shared-memory atomics, and passes over it
// again for the moments of N, of N_c and of the result.  Here h~ stays in its
// slab and the increments dN = sum +-W g go to a second one, so that
//   * one pass forms h_c = h~ + dN / w where a sample reached the node and sums
//     its moments (5 multiply-adds a node with tables of A v^k) and those of dN;
//   * the output moments follow from the 30 sums of degree <= 4 and mu
//     (lz_finish's formula), without a pass over the result;
//   * a shared sample set is applied without atomics: each thread sums its run
//     of the destination-sorted terms (k_scatter_*) in a register;
//   * per-cell sets need no storage per sample (products and node indices),
//     so two CTAs fit an SM where k_cell's 1024 threads had one.
// FP64 work per node falls from about 25 operations to 12, plus 5 on nodes
// that a sample reaches; GB300's FP64 pipe (about 2 a cycle and SM) bounds the
// FP64 cells.  Ten steps with a
// read-out, k_cell against k_relax: 16^2 x 12^3 FP64, 1000 samples, 1400 -> 668 us;
// 33 x 47 x 14^3 FP64 stretched, 3000 samples, 6467 -> 3885 us; four steps of 64^2 x
// 24^3 with 10^4 samples per cell (FP32) 10.73 -> 6.70 ms.
#pragma once

#include "bz_lazy.cuh"

#include <algorithm>

namespace bzk {

constexpr int kRxMaxN = 32;

template <typename R>
struct RxSmem {
    R *Av;                  // [5][N]: A v^k
    R *v, *v2, *IA, *cu, *ax, *cx;  // N each; ax: |Courant number| at the cell's width
    R *e0;                  // [32]: equilibrium sums of the 30 monomials
    R *part;                // [warps][32] partial sums; redraw queue of the per-cell sampler
    R *X, *D;               // [32] totals of N_c over the 30 monomials, [8] of dN
    R *Xl;                  // [32] rounding errors of X (FP32)
    R *mu;                  // [8]
    R *h, *d, *gw;          // slabs of h~ and dN; products of the shared set
    unsigned char *px;      // [5][16] lz_psiphi
};
template <typename R>
__host__ __device__ inline size_t rx_smem(RxSmem<R> *s, char *base, int N, int nvt, int T, int nt_gw)
{
    size_t off = 0;
    auto take = [&](size_t n) { size_t o = off; off += n * sizeof(R); return (R *)(base + o); };
    RxSmem<R> x;
    x.h = take((size_t)(nvt + 3) / 4 * 4);
    x.d = take((size_t)(nvt + 3) / 4 * 4);
    x.gw = take((size_t)nt_gw);
    off = (off + 15) & ~(size_t)15;
    x.Av = take(5 * N);
    x.v = take(N);
    x.v2 = take(N);
    x.IA = take(N);
    x.cu = take(N);
    x.ax = take(N);
    x.cx = take(N);
    x.e0 = take(32);
    x.part = take((size_t)(T / 32) * 32);
    x.X = take(32);
    x.D = take(8);
    x.Xl = take(sizeof(R) == 4 ? 32 : 0);
    x.mu = take(8);
    x.px = (unsigned char *)(base + off);
    off += 80;
    if (s) *s = x;
    return (off + 15) & ~(size_t)15;
}

// The 26 monomial sums from power sums s_p = sum n v_x^p at fixed (y, z).
template <typename R>
__device__ __forceinline__ void rx_mono(const R (&s)[5], R y, R z, R (&M)[32])
{
    const R y2 = y * y, z2 = z * z, q = y2 + z2, ys = y * s[0], zs = z * s[0], yzs = z * ys;
    M[0] = s[0];
    M[1] = s[1];
    M[2] = ys;
    M[3] = zs;
    M[4] = s[2];
    M[5] = y * ys;
    M[6] = z * zs;
    M[7] = y * s[1];
    M[8] = z * s[1];
    M[9] = yzs;
    M[10] = s[3];
    M[11] = y2 * ys;
    M[12] = z2 * zs;
    M[13] = y * s[2];
    M[14] = z * s[2];
    M[15] = y2 * s[1];
    M[16] = y * yzs;
    M[17] = z2 * s[1];
    M[18] = z * yzs;
    M[19] = y * M[8];
    const R t2 = s[2] + q * s[0], t3 = s[3] + q * s[1];
    M[20] = s[4] + q * s[2];
    M[21] = y2 * t2;
    M[22] = z2 * t2;
    M[23] = y * t3;
    M[24] = z * t3;
    M[25] = y * z * t2;
}

// A node that a sample reached (no FP64 comparison for doubles).
__device__ __forceinline__ bool rx_set(float x) { return x != 0.f; }
__device__ __forceinline__ bool rx_set(double x) { return __double_as_longlong(x) != 0; }

// Sums of 32 values over a warp by recursive halving: lane l gets value l.
template <typename R>
__device__ __forceinline__ R rx_reduce_scatter(R (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const R send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
    }
    return v[0];
}

// G mu = -D in FP64 by elimination (G is symmetric positive definite; one
// division a pivot), with the pivoted solve when a pivot is not positive.
// Every lane of the warp computes the same.
static __device__ __noinline__ void rx_solve_fallback(const Geo *g, const double *P, double *mu, int *fallback)
{
    correction_solve<double>(*g, P, mu, fallback);
}
__device__ __forceinline__ void rx_solve(const Geo &g, const double (&P)[19], double (&mu)[5], int *fallback)
{
    const double e = g.eps, p4 = P[4] + P[5] + P[6];
    const double m[5][5] = {{P[0], P[1], P[2], P[3], p4},
                            {P[1], P[4], P[7], P[8], P[10]},
                            {P[2], P[7], P[5], P[9], P[11]},
                            {P[3], P[8], P[9], P[6], P[12]},
                            {p4, P[10], P[11], P[12], P[13]}};
    double U[5][5], b[5], ip[5];
    bool ok = g.solve_fb == 0;
#pragma unroll
    for (int a = 0; a < 5; ++a) {
#pragma unroll
        for (int c = 0; c < 5; ++c) U[a][c] = g.G0[a * 5 + c] + e * m[a][c];
        b[a] = -P[14 + a];
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        ok = ok && U[k][k] > 0.0;
        ip[k] = 1.0 / U[k][k];
#pragma unroll
        for (int i = k + 1; i < 5; ++i) {
            const double f = U[i][k] * ip[k];
#pragma unroll
            for (int j = k + 1; j < 5; ++j) U[i][j] -= f * U[k][j];
            b[i] -= f * b[k];
        }
    }
    if (!ok) {
        double p[19], x[5];
#pragma unroll
        for (int k = 0; k < 19; ++k) p[k] = P[k];
        int f2 = 0;
        rx_solve_fallback(&g, p, x, &f2);
        if ((threadIdx.x & 31) == 0) *fallback += f2;
#pragma unroll
        for (int k = 0; k < 5; ++k) mu[k] = x[k];
        return;
    }
#pragma unroll
    for (int i = 4; i >= 0; --i) {
        double s = b[i];
#pragma unroll
        for (int j = i + 1; j < 5; ++j) s -= U[i][j] * mu[j];
        mu[i] = s * ip[i];
    }
}
__device__ __forceinline__ void rx_solve(const Geo &g, const float (&P)[19], float (&mu)[5], int *fallback)
{
    if (correction_spd(g, P, mu, threadIdx.x & 31)) return;
    lz_solve_fallback(g, P, mu);
    if ((threadIdx.x & 31) == 0) ++*fallback;
}

// Correction and moments of a cell (one warp): X holds the 26 sums of N_c and
// room for 30, D the sums of dN over 1, v_x, v_y, v_z, v^2.
template <typename R>
__device__ __forceinline__ void rx_finish(const Geo &g, const RxSmem<R> &S, double *mom, int *fallback)
{
    const int lane = threadIdx.x & 31;
    R *X = S.X;
    if (lane >= kLzMono && lane < kLzX) {
        const int i = lane - kLzMono;
        X[lane] = i == 0 ? X[4] + X[5] + X[6] : i == 1 ? X[10] + X[15] + X[17]
                  : i == 2 ? X[13] + X[11] + X[18] : X[14] + X[16] + X[12];
    }
    __syncwarp();
    R P[19], mu[5];
#pragma unroll
    for (int k = 0; k < 10; ++k) P[k] = X[k];
    P[10] = X[27];
    P[11] = X[28];
    P[12] = X[29];
    P[13] = X[20] + X[21] + X[22];
#pragma unroll
    for (int k = 0; k < 5; ++k) P[14 + k] = S.D[k];
    rx_solve(g, P, mu, fallback);
    if (lane < 5) {
        R m = mu[0];
#pragma unroll
        for (int k = 1; k < 5; ++k) m = lane == k ? mu[k] : m;
        S.mu[lane] = m;
    }
    if (!mom) return;
    if constexpr (sizeof(R) == 4) {
        lz_moments(X, S.Xl, S.e0, S.px, mu, g.epsf, mom);
        return;
    }
    const R eps = (R)g.eps;
    R m = R(0);
    if (lane < 10) {
        // sum w h phi = sum N_c phi + sum_a mu_a (E0 + eps sum N_c psi_a phi)
        m = X[lane];
#pragma unroll 1
        for (int k = 0; k < 5; ++k) {
            const int x = S.px[k * 16 + lane];
            m += S.mu[k] * (S.e0[x] + eps * X[x]);
        }
    }
    const unsigned all = 0xFFFFFFFFu;
    const R rho = __shfl_sync(all, m, 0), n = R(1) + eps * rho;
    const R u0 = __shfl_sync(all, m, 1) / n, u1 = __shfl_sync(all, m, 2) / n, u2 = __shfl_sync(all, m, 3) / n;
    const R tr = __shfl_sync(all, m, 4) + __shfl_sync(all, m, 5) + __shfl_sync(all, m, 6);
    const R mq = __shfl_sync(all, m, lane - 1 & 31);
    const R ua = lane == 5 || lane == 8 || lane == 9 ? u0 : lane == 6 || lane == 10 ? u1 : u2;
    const R ub = lane == 5 ? u0 : lane == 6 || lane == 8 ? u1 : u2;
    R o = R(2) * mq - R(2) * eps * n * ua * ub;
    if (lane == 0) o = rho;
    if (lane == 1) o = u0;
    if (lane == 2) o = u1;
    if (lane == 3) o = u2;
    if (lane == 4) o = ((R(2) / R(3)) * tr - rho) / n - (R(2) * eps / R(3)) * (u0 * u0 + u1 * u1 + u2 * u2);
    if (lane < 11) mom[lane] = (double)o;
}

// Terms of a shared set sorted by destination: entry = node << 17 | loss <<
// 16 | sample (samples below 65536, nodes below 32768), C entries a thread at
// stride T (meta: the number of entries, C).

// The shared sample sets of K consecutive steps, built in one launch per
// kernel: step n in slot n mod K.  (Per step, the FP64 draw of the set alone
// is a 40 us chain on the critical path of a small cavity's 140 us step.)
template <typename R> struct RxPlans {
    int K, nt, nvt, T;
    PlanA<R, uint16_t> *pa;         // K x nt: (a, b, W)
    ushort4 *idx;                   // K x nt: the four nodes
    int *count, *cursor;            // K x nvt
    int *meta;                      // K x 2
    uint32_t *ent;                  // K x entn
    int64_t entn;
    unsigned long long *cnt;        // K x 2: samples with a node outside the box, near a face
};
template <typename R>
__global__ void k_rx_plan(Geo g, RxPlans<R> A, int64_t step0)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t step = step0 + blockIdx.y;
    const int s = (int)(step % A.K);
    const bool act = l < A.nt;
    SampleOut o = {};
    if (act) {
        o = draw_sample(g, step, 0xFFFFFFFFu, (uint32_t)l);
        A.idx[(int64_t)s * A.nt + l] = Idx4<uint16_t>::make(o.idx);
        A.pa[(int64_t)s * A.nt + l] = make_plan_a<R, uint16_t>(o.idx[0], o.idx[1], o.W);
        int *c = A.count + (int64_t)s * A.nvt;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (o.idx[k] >= 0) atomicAdd(c + o.idx[k], 1);
    }
    const unsigned mo = __ballot_sync(0xFFFFFFFFu, act && o.outside);
    const unsigned mn = __ballot_sync(0xFFFFFFFFu, act && o.near);
    if ((threadIdx.x & 31) == 0) {
        if (mo) atomicAdd(A.cnt + 2 * s, (unsigned long long)__popc(mo));
        if (mn) atomicAdd(A.cnt + 2 * s + 1, (unsigned long long)__popc(mn));
    }
}
template <typename R>
__global__ void __launch_bounds__(1024) k_rx_scan(RxPlans<R> A, int64_t step0)
{
    __shared__ int part[1024];
    const int s = (int)((step0 + blockIdx.x) % A.K);
    const int64_t v = (int64_t)s * A.nvt;
    scatter_scan_body(A.nvt, A.T, A.count + v, A.cursor + v, A.meta + 2 * s, part);
}
template <typename R>
__global__ void k_rx_fill(RxPlans<R> A, int64_t step0)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= A.nt) return;
    const int s = (int)((step0 + blockIdx.y) % A.K);
    const int C = A.meta[2 * s + 1];
    const ushort4 q = A.idx[(int64_t)s * A.nt + l];
    const unsigned short d[4] = {q.x, q.y, q.z, q.w};
    int *cur = A.cursor + (int64_t)s * A.nvt;
    uint32_t *ent = A.ent + s * A.entn;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (d[k] == 0xFFFF) continue;
        const int pos = atomicAdd(cur + d[k], 1), tt = pos / C;
        ent[(int64_t)(pos - tt * C) * A.T + tt] = (uint32_t)d[k] << 17 | (k < 2 ? 0x10000u : 0u) | (uint32_t)l;
    }
}
// End of a step: the sample counts of its plan, and the step counter.
static __global__ void k_rx_advance(int64_t *__restrict__ stepp, int K, const unsigned long long *__restrict__ cnt,
                                    unsigned long long *__restrict__ stats)
{
    const int s = (int)(*stepp % K);
    stats[1] += cnt[2 * s];
    stats[2] += cnt[2 * s + 1];
    *stepp += 1;
}

// A thread's run of n sorted terms in FP32.  A finished node is one predicated store
// (a branch per node keeps the lanes of a warp apart at nearly every term); the first
// node's sum goes to the thread's slot, and it and the last one, which neighbouring
// runs may share, are added atomically at the end.  Four terms are in flight while
// the previous four are summed (eight: 667 us where four take 632, by spills).
__device__ __forceinline__ void rx_step(uint32_t w, float r, uint32_t base, uint32_t &prev, uint32_t &p, float &acc)
{
    asm volatile("{\n .reg .pred q;\n .reg .b32 x;\n xor.b32 x, %3, %2;\n setp.ge.u32 q, x, 0x20000;\n"
                 " @q st.shared.f32 [%0], %1;\n shr.u32 x, %3, 17;\n @q mad.lo.u32 %0, x, 4, %5;\n"
                 " @q mov.f32 %1, 0f00000000;\n add.rn.f32 %1, %1, %4;\n}"
                 : "+r"(p), "+f"(acc) : "r"(prev), "r"(w), "f"(r), "r"(base) : "memory");
    prev = w;
}
__device__ __forceinline__ void rx_run(int n, const uint32_t *__restrict__ list, int T, float *d, float *slot, const float *gw)
{
    if (n <= 0) return;
    const uint32_t base = lz_saddr(d), sl = lz_saddr(slot);
    auto val = [&](uint32_t w) {
        return __uint_as_float(__float_as_uint(gw[w & 0xFFFFu]) ^ (w << 15 & 0x80000000u));
    };
    uint32_t e[4], f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) e[u] = list[(int64_t)min(u, n - 1) * T];
    const uint32_t first = e[0];
    uint32_t prev = first, p = sl;
    float acc = 0.f;
    int i = 0;
    for (; i + 4 < n; i += 4) {
        float r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) f[u] = list[(int64_t)min(i + 4 + u, n - 1) * T];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = val(e[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) rx_step(e[u], r[u], base, prev, p, acc);
#pragma unroll
        for (int u = 0; u < 4; ++u) e[u] = f[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (i + u < n) rx_step(e[u], val(e[u]), base, prev, p, acc);
    atomicAdd(d + (prev >> 17), acc);
    if (p != sl) atomicAdd(d + (first >> 17), *slot);
}

// Threads of a CTA for a shared set: those of the columns, and in FP32 (64 registers a
// thread) as many more as its share of an SM has room for, which help with the samples
// and the sorted terms, from 0.3 times as many samples as nodes.  64^2 cells, us with the
// columns' threads / with more, at 0.1, 0.25, 0.35 and 0.8 samples per node: 24^3
// 468 / 477, 517 / 521, 558 / 545, 714 / 664; 20^3 264 / 265, 291 / 291, 310 / 308, 391 /
// 378; 21^3 286 / 289, 317 / 319, 335 / 338, 418 / 418; up to 16^3 the CTAs that share
// an SM leave no room for more.
template <typename R>
inline int rx_threads(int N, int nvt, int nseg, int nt, size_t smem_sm)
{
    const int T = (N * N * nseg + 31) / 32 * 32;
    if (sizeof(R) == 8 || 10 * nt < 3 * nvt) return T;
    const size_t need = rx_smem<R>(nullptr, nullptr, N, nvt, kMaxThreads, nt) + 1024;
    const int ctas = (int)(smem_sm / need);
    return ctas < 1 ? T : std::max(T, kMaxThreads / ctas / 32 * 32);
}

// FUSED: h~ by streaming hin, else h~ = hin.  PC: the cell's own sample set.
// A thread owns the column (jy, jz) = p of a segment of jx: items i = p + N^2
// seg, t = i (T >= N^2 nseg).
template <typename R, bool FUSED, bool PC, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
k_relax(const __grid_constant__ Geo g, int nseg, const R *__restrict__ hin, const R *__restrict__ ghost,
        RxPlans<R> A, R *__restrict__ hout, double *__restrict__ mom,
        unsigned long long *__restrict__ stats, const int64_t *__restrict__ stepp)
{
    extern __shared__ __align__(16) char smem_raw[];
    const int N = g.nv, N2 = N * N, nvt = g.nvt, T = blockDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    RxSmem<R> S;
    rx_smem<R>(&S, smem_raw, N, nvt, T, PC ? 0 : g.nt);
    const R eps = (R)g.eps;
    const int64_t step = *stepp;
    const int slot = PC ? 0 : (int)(step % A.K);
    const PlanA<R, uint16_t> *pa = A.pa + (int64_t)slot * A.nt;
    const uint32_t *ent = A.ent + slot * A.entn;
    const int E = PC ? 0 : A.meta[2 * slot], C = PC ? 0 : A.meta[2 * slot + 1];
    for (int i = t; i < N; i += T) {
        const double v = g.axv[i], A = g.axA[i];
        double x = A;
        for (int k = 0; k < 5; ++k) {
            S.Av[k * N + i] = (R)x;
            x *= v;
        }
        S.v[i] = (R)v;
        S.v2[i] = (R)(v * v);
        S.IA[i] = (R)(1.0 / A);
        S.cu[i] = (R)(v * g.dt / g.dx);
    }
    if (t < 32) {
        // The equilibrium sum of monomial t: a product of axis sums E_k = sum
        // A v^k (lane k < 5 holds E_k), or for those with v^2 a sum of three.
        double Ek = 0.0;
        if (t < 5)
            for (int i = 0; i < N; ++i) {
                double x = g.axA[i];
                for (int k = 0; k < t; ++k) x *= g.axv[i];
                Ek += x;
            }
        double E[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) E[k] = __shfl_sync(0xFFFFFFFFu, Ek, k);
        S.e0[t] = (R)lz_equilibrium(t, E);
    }
    for (int i = t; i < 50; i += T) S.px[i / 10 * 16 + i % 10] = (unsigned char)lz_psiphi(i / 10, i % 10);
    // The thread's column and its range of jx.
    const bool col = t < N2 * nseg;
    const int cwarps = (N2 * nseg + 31) / 32;        // (the other warps help with the samples)
    const int seg = col ? t / N2 : 0, p = col ? t - seg * N2 : 0, jy = p / N, jz = p - jy * N;
    const int x0 = seg * N / nseg, x1 = (seg + 1) * N / nseg;
    const int nneg = N / 2, npos = (N + 1) / 2;
    int fallback = 0;
    __syncthreads();
    const R ry = (R)(g.dx / g.dy);
    const R vy = S.v[jy], vz = S.v[jz], Ayz = S.Av[jy] * S.Av[jz], IAyz = S.IA[jy] * S.IA[jz];

    for (int kc = blockIdx.x; kc < g.nr; kc += gridDim.x) {
        const int c = cell_of(g, kc), ix = c % g.nx, iy = c / g.nx;
        const R *own = hin + (int64_t)c * nvt;
        if (FUSED) {
            const R fx = g.sx ? (R)g.sx[ix] : R(1);
            for (int i = t; i < N; i += T) S.ax[i] = fabs(S.cu[i]) * fx;
            __syncthreads();
        }
        // ---- h~, and dN = 0
        if (col) {
            R ay = R(0);
            const R *ys = own, *xr = own, *xl = own;
            int ystr = N2, yoff = p, rstr = N2, lstr = N2, ro = p, lo = p;
            if (FUSED) {
                const R fy = g.sy ? (R)g.sy[iy] : ry;
                ay = fabs(S.cu[jy]) * fy;
                if (vy > R(0)) {
                    if (iy > 0) ys = own - (int64_t)g.nx * nvt;
                    else { ys = ghost + (2 * g.ny + ix) * N; ystr = 1; yoff = 0; }
                } else if (vy < R(0)) {
                    if (iy < g.ny - 1) ys = own + (int64_t)g.nx * nvt;
                    else { ys = ghost + (2 * g.ny + g.nx + ix) * N; ystr = 1; yoff = 0; }
                }
                if (ix < g.nx - 1) xr = own + nvt;
                else { xr = ghost + (g.ny + iy) * N + jy; rstr = 0; ro = 0; }
                if (ix > 0) xl = own - nvt;
                else { xl = ghost + iy * N + jy; lstr = 0; lo = 0; }
            }
#pragma unroll 4
            for (int jx = x0; jx < x1; ++jx) {
                const int j = jx * N2 + p;
                R h = own[j];
                if (FUSED) {
                    const R hx = jx < nneg ? xr[jx * rstr + ro] : jx >= npos ? xl[jx * lstr + lo] : h;
                    const R hy = ys[jx * ystr + yoff];
                    h = h - S.ax[jx] * (h - hx) - ay * (h - hy);
                }
                S.h[j] = h;
                S.d[j] = R(0);
            }
        }
        if (PC && t == 0) reinterpret_cast<int *>(S.part)[0] = 0;
        __syncthreads();

        // ---- the collision increments (Eq. monteCarloInt on h~)
        if constexpr (PC) {
            const bool fast = sizeof(R) == 4 && !g.axe;
            int *rq = reinterpret_cast<int *>(S.part);
            const int room = (T / 32) * 32 * (int)(sizeof(R) / 4) - 1;
            const int rcap = g.redraw_cap < 0 ? room : min(g.redraw_cap, room);
            auto put = [&](const SampleOut &o, R W) {
                const R ha = o.idx[0] >= 0 ? S.h[o.idx[0]] : R(0), hb = o.idx[1] >= 0 ? S.h[o.idx[1]] : R(0);
                const R r = (ha + hb * (R(1) + eps * ha)) * W;
                if (r == R(0)) return;
                if (o.idx[2] >= 0) atomicAdd(S.d + o.idx[2], r);
                if (o.idx[3] >= 0) atomicAdd(S.d + o.idx[3], r);
                if (o.idx[0] >= 0) atomicAdd(S.d + o.idx[0], -r);
                if (o.idx[1] >= 0) atomicAdd(S.d + o.idx[1], -r);
            };
            auto count = [&](bool act, const SampleOut &o) {
                if (stats) {
                    const unsigned mo = __ballot_sync(0xFFFFFFFFu, act && o.outside);
                    const unsigned mn = __ballot_sync(0xFFFFFFFFu, act && o.near);
                    if (lane == 0) {
                        if (mo) atomicAdd(stats + 1, (unsigned long long)__popc(mo));
                        if (mn) atomicAdd(stats + 2, (unsigned long long)__popc(mn));
                    }
                }
            };
            // A sample near a velocity-cell face is queued and drawn again in
            // FP64 (draw_sample_fast); a full queue draws in place.
            for (int l0 = 0; l0 < g.nt; l0 += T) {
                const int l = l0 + t;
                bool act = l < g.nt;
                SampleOut o = {};
                if (act) {
                    bool redo = true;
                    float Wf = 0.f;
                    if (fast) o = draw_sample_fast(g, step, (uint32_t)c, (uint32_t)l, &redo, &Wf);
                    if (redo) {
                        const int k = fast ? atomicAdd(rq, 1) : rcap;
                        if (k < rcap) {
                            rq[1 + k] = l;
                            act = false;
                        } else {
                            o = draw_sample(g, step, (uint32_t)c, (uint32_t)l);
                        }
                    }
                    if (act) put(o, redo ? (R)o.W : (R)Wf);
                }
                count(act, o);
            }
            if (fast) {
                __syncthreads();
                const int nq = min(rq[0], rcap);
                for (int i0 = 0; i0 < nq; i0 += T) {
                    const bool act = i0 + t < nq;
                    SampleOut o = {};
                    if (act) {
                        o = draw_sample(g, step, (uint32_t)c, (uint32_t)rq[1 + i0 + t]);
                        put(o, (R)o.W);
                    }
                    count(act, o);
                }
            }
        } else {
            for (int l = t; l < g.nt; l += T) {
                const PlanA<R, uint16_t> q = pa[l];
                const int a = q.a(), b = q.b();
                const R ha = a >= 0 ? S.h[a] : R(0), hb = b >= 0 ? S.h[b] : R(0);
                S.gw[l] = (ha + hb * (R(1) + eps * ha)) * q.W;
            }
            __syncthreads();
            // Each thread's run of the sorted terms: a destination's sum is
            // stored when the next one begins; the run's first and last
            // destination may be shared with a neighbour (atomically).
            const int n = min(C, E - t * C);
            if constexpr (sizeof(R) == 4) {
                rx_run(n, ent + t, T, S.d, S.part + t, S.gw);
            } else {
                R acc = R(0);
                int cur = -1;
                bool first = true;
                auto flush = [&]() {
                    if (first) atomicAdd(S.d + cur, acc);
                    else S.d[cur] = acc;
                    first = false;
                };
                for (int i0 = 0; i0 < n; i0 += 4) {
                    uint32_t e[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) e[u] = i0 + u < n ? ent[(int64_t)(i0 + u) * T + t] : 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (i0 + u >= n) break;
                        const int node = (int)(e[u] >> 17);
                        const R r = S.gw[e[u] & 0xFFFFu];
                        if (node != cur) {
                            if (cur >= 0) flush();
                            cur = node;
                            acc = R(0);
                        }
                        acc += e[u] & 0x10000u ? -r : r;
                    }
                }
                if (cur >= 0) atomicAdd(S.d + cur, acc);
            }
        }
        __syncthreads();

        // ---- h_c = h~ + dN / w, the sums of dN and of N_c = w h_c, the correction
        R M[32];
        {
            R s[5] = {R(0), R(0), R(0), R(0), R(0)}, d0 = R(0), d1 = R(0), d2 = R(0);
            if (col) {
#pragma unroll 2
                for (int jx = x0; jx < x1; ++jx) {
                    const int j = jx * N2 + p;
                    const R x = S.d[j];
                    R h = S.h[j];
                    if (rx_set(x)) {
                        h += (x * IAyz) * S.IA[jx];
                        S.h[j] = h;
                        d0 += x;
                        d1 += x * S.v[jx];
                        d2 += x * S.v2[jx];
                    }
#pragma unroll
                    for (int k = 0; k < 5; ++k) s[k] += S.Av[k * N + jx] * h;
                }
#pragma unroll
                for (int k = 0; k < 5; ++k) s[k] *= Ayz;
            }
            rx_mono(s, vy, vz, M);
            M[26] = d0;
            M[27] = d1;
            M[28] = vy * d0;
            M[29] = vz * d0;
            M[30] = d2 + (vy * vy + vz * vz) * d0;
            M[31] = R(0);
        }
        if (warp < cwarps) S.part[warp * 32 + lane] = rx_reduce_scatter(M);
        __syncthreads();
        if (warp == 0) {
            R tot = R(0);
            if constexpr (sizeof(R) == 4) {
                float f = 0.f, fc = 0.f;                 // compensated
                for (int w = 0; w < cwarps; ++w) {
                    float e;
                    two_sum(f, S.part[w * 32 + lane], f, e);
                    fc = __fadd_rn(fc, e);
                }
                float lo;
                two_sum(f, fc, tot, lo);
                S.Xl[lane] = lo;
            } else {
                for (int w = 0; w < cwarps; ++w) tot += S.part[w * 32 + lane];
            }
            if (lane < kLzMono) S.X[lane] = tot;
            else if (lane < 31) S.D[lane - kLzMono] = tot;
            __syncwarp();
            rx_finish<R>(g, S, mom ? mom + (int64_t)c * 11 : nullptr, &fallback);
            __syncwarp();
            for (int i = lane; i < N; i += 32) S.cx[i] = S.mu[1] * S.v[i] + S.mu[4] * (S.v[i] * S.v[i]);
        }
        __syncthreads();

        // ---- the corrected result
        if (col) {
            const R ct = S.mu[0] + S.mu[2] * vy + S.mu[3] * vz + S.mu[4] * (vy * vy + vz * vz);
            R *dst = hout + (int64_t)c * nvt;
#pragma unroll 4
            for (int jx = x0; jx < x1; ++jx) {
                const int j = jx * N2 + p;
                const R h = S.h[j], kap = ct + S.cx[jx];
                dst[j] = h + (R(1) + eps * h) * kap;
            }
        }
        __syncthreads();
    }
    if (fallback && stats) atomicAdd(stats + 3, (unsigned long long)fallback);
}

}  // namespace bzk
