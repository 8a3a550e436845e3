// bz_cell4.cuh -- per-cell relaxation kernel, FP32 fast path.
//
// Same mathematics as k_cell (Eqs. streaming2D, monteCarloInt,
// collision_step, rinorm_a, correzione, densita..sforzi) for FP32 states whose
// velocity axis has a multiple of 4 nodes.  Thread t owns a "quad" of four
// consecutive jz nodes of one (jy) row and a contiguous range of J jx-planes:
//   q = t mod Q (Q = N^2/4 quads per plane), k = t div Q, jx in [kJ, kJ + J).
// All slab traffic (global and shared) is 16-byte vectors and the per-jx
// tables are read as broadcast float4s shared by the quad's four nodes.  The
// scatter of Eq. monteCarloInt walks a destination-sorted list of the step's
// terms (built once per step by k_scatter_*), so a thread adds the sum of a
// node's terms with one shared-memory atomic instead of one per term.
#pragma once

#include "bz_kernels.cuh"

namespace bzk {

constexpr int kClkCells = 8;    // cells traced per launch (CTA 0)
constexpr int kClkPhases = 9;   // stamps per cell

struct Map4 {
    int Q;   // quads per jx-plane (N^2 / 4)
    int K;   // jx chunks
    int J;   // jx planes per chunk (N / K)
};

// Shared-memory layout of k_cell4.
struct Cell4Smem {
    float *red;      // kMaxWarps * 32
    double *tot;     // 32 (totf aliases its first 128 bytes)
    double *mu;      // 8
    float4 *conv;    // N: {A, v, v^2, 0}
    float4 *gram;    // N: {v, v^2, v^3, v^4}
    float4 *fin;     // N: {1/A, cx, A, A v}   (cx = mu_x v + mu_4 v^2, per cell)
    float *Av2;      // N: A v^2
    float *cu;       // N: v dt/dx
    float *v;        // N
    float *A;        // N
    float *IA;       // N
    int *rot;        // N: jx mod (N/4), the quad rotation of plane jx
    float4 *vzq;     // N/4: v of the four jz nodes of quad column qz
    float4 *Azq;     // N/4: A of those nodes
    float4 *IAzq;    // N/4: 1/A of those nodes
    float4 *slab4;   // N^3 / 4
    float *gw;       // Nt: g_l W_l of the gather phase
};

__host__ __device__ inline size_t cell4_smem_bytes(int nv, int nvt, int nt)
{
    size_t off = sizeof(float) * kMaxWarps * 32 + sizeof(double) * (32 + 8);
    off += sizeof(float4) * 3 * nv + sizeof(float) * 5 * nv + sizeof(int) * nv;
    off = (off + 15) & ~(size_t)15;
    off += sizeof(float4) * 3 * (nv / 4);
    off += sizeof(float) * nvt;
    off += sizeof(float) * nt;
    return off;
}

__device__ __forceinline__ Cell4Smem carve4(char *base, int N, int nvt)
{
    Cell4Smem s;
    size_t off = 0;
    s.red = (float *)(base + off); off += sizeof(float) * kMaxWarps * 32;
    s.tot = (double *)(base + off); off += sizeof(double) * 32;
    s.mu = (double *)(base + off); off += sizeof(double) * 8;
    s.conv = (float4 *)(base + off); off += sizeof(float4) * N;
    s.gram = (float4 *)(base + off); off += sizeof(float4) * N;
    s.fin = (float4 *)(base + off); off += sizeof(float4) * N;
    s.Av2 = (float *)(base + off); off += sizeof(float) * N;
    s.cu = (float *)(base + off); off += sizeof(float) * N;
    s.v = (float *)(base + off); off += sizeof(float) * N;
    s.A = (float *)(base + off); off += sizeof(float) * N;
    s.IA = (float *)(base + off); off += sizeof(float) * N;
    s.rot = (int *)(base + off); off += sizeof(int) * N;
    off = (off + 15) & ~(size_t)15;
    s.vzq = (float4 *)(base + off); off += sizeof(float4) * (N / 4);
    s.Azq = (float4 *)(base + off); off += sizeof(float4) * (N / 4);
    s.IAzq = (float4 *)(base + off); off += sizeof(float4) * (N / 4);
    s.slab4 = (float4 *)(base + off);
    off += sizeof(float) * nvt;
    s.gw = (float *)(base + off);
    return s;
}

// Destination-sorted scatter list of a step (shared by every cell): every
// valid (node, sample, sign) term of Eq. monteCarloInt as one 32-bit word
// node << 16 | loss << 15 | l, sorted by node by a counting sort, and stored
// so that thread t of the cell kernel reads its contiguous run of C words at
// stride T (coalesced).  meta[0] = number of words E, meta[1] = C.
static __global__ void k_scatter_count(int nt, const ushort4 *__restrict__ pidx, int *__restrict__ count)
{
    int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nt) return;
    ushort4 q = pidx[l];
    if (q.x != 0xFFFF) atomicAdd(count + q.x, 1);
    if (q.y != 0xFFFF) atomicAdd(count + q.y, 1);
    if (q.z != 0xFFFF) atomicAdd(count + q.z, 1);
    if (q.w != 0xFFFF) atomicAdd(count + q.w, 1);
}

// Exclusive scan of the per-node counts (one CTA of 1024 threads).
// gate (nullable): when it is given and gate[1] is 0, the kernel does nothing.
// Exclusive scan of the per-node counts (one CTA of 1024 threads, part: 1024
// ints of shared memory): cursor = first position of each node's words,
// meta = {E, C = ceil(E / T)}.
__device__ __forceinline__ void scatter_scan_body(int nvt, int T, const int *__restrict__ count,
                                                  int *__restrict__ cursor, int *__restrict__ meta,
                                                  int *part)
{
    const int t = threadIdx.x, per = (nvt + 1023) / 1024;
    const int b = t * per, e = min(nvt, b + per);
    int s = 0;
    for (int j = b; j < e; ++j) s += count[j];
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {       // Hillis-Steele inclusive scan
        int v = t >= off ? part[t - off] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int run = part[t] - s;
    for (int j = b; j < e; ++j) {
        cursor[j] = run;
        run += count[j];
    }
    if (t == 1023) {
        meta[0] = part[1023];
        meta[1] = (part[1023] + T - 1) / T;
    }
}

static __global__ void __launch_bounds__(1024) k_scatter_scan(int nvt, int T, const int *__restrict__ count,
                                                      int *__restrict__ cursor, int *__restrict__ meta,
                                                      const int *__restrict__ gate = nullptr)
{
    if (gate && !gate[1]) return;
    __shared__ int part[1024];
    scatter_scan_body(nvt, T, count, cursor, meta, part);
}

static __global__ void k_scatter_fill(int nt, int T, const ushort4 *__restrict__ pidx,
                               int *__restrict__ cursor, const int *__restrict__ meta,
                               uint32_t *__restrict__ ent, const int *__restrict__ gate = nullptr)
{
    if (gate && !gate[1]) return;
    int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nt) return;
    const int C = meta[1];
    const ushort4 q = pidx[l];
    const unsigned short d[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (d[k] == 0xFFFF) continue;
        const int pos = atomicAdd(cursor + d[k], 1);
        const int tt = pos / C, i = pos - tt * C;
        ent[(int64_t)i * T + tt] = ((uint32_t)d[k] << 16) | (k < 2 ? 0x8000u : 0u) | (uint32_t)l;
    }
}

// G mu = -D (Eqs. rinorm_a, correzione): the correction restores the
// conserved moments of h~, so its right-hand side is minus the conserved
// moments of the collision increment, D_a = sum_j psi_a (N_c,j - N_j), taken
// directly from the increment sums (never as the difference of the large
// post- and pre-collision sums).  P[0..13] are the moment sums of N_c over
// 1, vx, vy, vz, vx2, vy2, vz2, vxvy, vxvz, vyvz, vx v2, vy v2, vz v2, v4
// (they give G = G0 + eps sum_j N_c psi psi^T) and P[14..18] the increment
// sums D over 1, vx, vy, vz, v2.  Solved in registers by Gaussian
// elimination without pivoting (stable for the symmetric positive definite
// Gram matrix), then one step of iterative refinement whose residual
// -D - G mu is evaluated exactly with error-free products and sums and
// rounded once, so mu is as accurate as the FP32 entries of G and D allow.
// False if a pivot is not positive.  lane >= 0: all 32 lanes of a warp call
// it with the same P and their lane index, and lane a < 5 evaluates row a of
// the residual (the rest is the same on every lane).
__device__ __forceinline__ bool correction_spd(const Geo &g, const float *P, float *mu, int lane = -1)
{
    if (g.solve_fb) return false;
    const float e = g.epsf;
    const float p4 = P[4] + P[5] + P[6];
    const float m[5][5] = {
        {P[0], P[1], P[2], P[3], p4},
        {P[1], P[4], P[7], P[8], P[10]},
        {P[2], P[7], P[5], P[9], P[11]},
        {P[3], P[8], P[9], P[6], P[12]},
        {p4, P[10], P[11], P[12], P[13]}};
    float A[5][5], U[5][5], L[5][5], ip[5], b[5], x[5];
#pragma unroll
    for (int a = 0; a < 5; ++a) {
#pragma unroll
        for (int c = 0; c < 5; ++c) A[a][c] = U[a][c] = g.G0f[a * 5 + c] + e * m[a][c];
        b[a] = -P[14 + a];
    }
#pragma unroll
    for (int kk = 0; kk < 5; ++kk) {
        const float piv = U[kk][kk];
        if (!(piv > 0.f)) return false;
        ip[kk] = 1.f / piv;
#pragma unroll
        for (int i = kk + 1; i < 5; ++i) {
            L[i][kk] = U[i][kk] * ip[kk];
#pragma unroll
            for (int j = kk + 1; j < 5; ++j) U[i][j] -= L[i][kk] * U[kk][j];
        }
    }
    // x = U^-1 L^-1 r, for the right-hand side and then the residual.
    auto lu_solve = [&](float (&r)[5], float (&y)[5]) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            float s = r[i];
#pragma unroll
            for (int k = 0; k < i; ++k) s -= L[i][k] * r[k];
            r[i] = s;
        }
#pragma unroll
        for (int i = 4; i >= 0; --i) {
            float s = r[i];
#pragma unroll
            for (int j = i + 1; j < 5; ++j) s -= U[i][j] * y[j];
            y[i] = s * ip[i];
        }
    };
    float r[5];
#pragma unroll
    for (int a = 0; a < 5; ++a) r[a] = b[a];
    lu_solve(r, x);
    // Row a of b - A x, exactly, rounded once.
    auto residual = [&](const float (&Ar)[5], float ba) {
        float hi = ba, lo = 0.f;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            float p, pe, s, se;
            two_prod(Ar[c], x[c], p, pe);
            two_sum(hi, -p, s, se);
            hi = s;
            lo = __fadd_rn(lo, __fsub_rn(se, pe));
        }
        return __fadd_rn(hi, lo);
    };
    if (lane < 0) {
#pragma unroll
        for (int a = 0; a < 5; ++a) r[a] = residual(A[a], b[a]);
    } else {
        float Ar[5], ba = 0.f;
#pragma unroll
        for (int c = 0; c < 5; ++c) Ar[c] = 0.f;
#pragma unroll
        for (int a = 0; a < 5; ++a)
            if (lane == a) {
#pragma unroll
                for (int c = 0; c < 5; ++c) Ar[c] = A[a][c];
                ba = b[a];
            }
        const float ra = residual(Ar, ba);
#pragma unroll
        for (int a = 0; a < 5; ++a) r[a] = __shfl_sync(0xFFFFFFFFu, ra, a);
    }
    float dx[5];
    lu_solve(r, dx);
#pragma unroll
    for (int a = 0; a < 5; ++a) mu[a] = x[a] + dx[a];
    return true;
}

// Sum K (<= 32) per-thread values over the block.  Inside a warp the values
// are transposed while being added (31 shuffles for any K <= 32, lane i ends
// with the warp total of value i); one thread per value then adds the warp
// totals.  Totals are stored in tot[0..K).
template <int K>
__device__ __forceinline__ void block_reduce4(float (&v)[K], float *red, float *tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i < K ? v[i] : 0.f;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            float send = up ? x[i] : x[i + w];
            float keep = up ? x[i + w] : x[i];
            x[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, w);
        }
    }
    if (lane < K) red[warp * 32 + lane] = x[0];
    __syncthreads();
    if (threadIdx.x < K) {
        // Compensated sum of the warp totals.
        float s = 0.f, c = 0.f;
        for (int w = 0; w < nwarps; ++w) {
            float e;
            two_sum(s, red[w * 32 + threadIdx.x], s, e);
            c = __fadd_rn(c, e);
        }
        tot[threadIdx.x] = __fadd_rn(s, c);
    }
    __syncthreads();
}

__device__ __forceinline__ float4 f4(float a) { return make_float4(a, a, a, a); }

// One upwind update of a quad (Eq. streaming2D, both signs handled by |Cu|).
__device__ __forceinline__ float4 upwind4(float4 h0, float4 hx, float4 hy, float ax, float ay)
{
    float4 o;
    o.x = h0.x - ax * (h0.x - hx.x) - ay * (h0.x - hy.x);
    o.y = h0.y - ax * (h0.y - hx.y) - ay * (h0.y - hy.y);
    o.z = h0.z - ax * (h0.z - hx.z) - ay * (h0.z - hy.z);
    o.w = h0.w - ax * (h0.w - hx.w) - ay * (h0.w - hy.w);
    return o;
}

// Free streaming alone (Eq. streaming2D) for FP32 states with a multiple-of-4
// velocity axis: each thread moves 16-byte quads of four jz nodes, one CTA
// per cell at a time in the strip order, interior cells without branches.
// SX: stretched cells (the cell's own widths scale its Courant numbers).
template <bool SX>
__global__ void __launch_bounds__(1024) k_stream4(Geo g, const float *__restrict__ hin,
                                                  const float *__restrict__ ghost,
                                                  float *__restrict__ hout)
{
    // blockDim.x is a multiple of Q: thread t keeps quad q = t mod Q of every
    // plane and walks the planes jx = t div Q, t div Q + blockDim.x / Q, ...
    __shared__ float scu[kMaxN];
    const int N = g.nv, nq = N / 4, Q = N * N / 4, half = N / 2;
    for (int i = threadIdx.x; i < N; i += blockDim.x) scu[i] = (float)(g.axv[i] * g.dt / g.dx);
    __syncthreads();
    const int64_t plane = g.nvt / 4;
    const float ry = (float)(g.dx / g.dy);
    const int q = threadIdx.x % Q, jxs = threadIdx.x / Q, jstep = blockDim.x / Q;
    const int jy = q / nq;
    float ay = fabsf(scu[jy] * ry), fx = 1.f;
    for (int kc = blockIdx.x; kc < g.nr; kc += gridDim.x) {
        const int c = cell_of(g, kc);
        const int ix = c % g.nx, iy = c / g.nx;
        if (SX) {
            // Courant factors of this cell: its own widths.
            fx = (float)g.sx[ix];
            ay = fabsf(scu[jy]) * (float)g.sy[iy];
        }
        const float4 *own = reinterpret_cast<const float4 *>(hin) + (int64_t)c * plane;
        float4 *dst = reinterpret_cast<float4 *>(hout) + (int64_t)c * plane;
        if (ix > 0 && ix < g.nx - 1 && iy > 0 && iy < g.ny - 1) {
            const float4 *ys = jy < half ? own + (int64_t)g.nx * plane : own - (int64_t)g.nx * plane;
            const float4 *xr = own + plane, *xl = own - plane;
#pragma unroll 4
            for (int jx = jxs; jx < N; jx += jstep) {
                const int o = jx * Q + q;
                const float4 hx = jx < half ? xr[o] : xl[o];
                dst[o] = upwind4(own[o], hx, ys[o], SX ? fabsf(scu[jx]) * fx : fabsf(scu[jx]), ay);
            }
        } else {
            for (int jx = jxs; jx < N; jx += jstep) {
                const int o = jx * Q + q;
                float4 hx, hy;
                if (jx < half) hx = ix < g.nx - 1 ? own[o + plane] : f4(ghost[(g.ny + iy) * N + jy]);
                else hx = ix > 0 ? own[o - plane] : f4(ghost[iy * N + jy]);
                if (jy < half)
                    hy = iy < g.ny - 1 ? own[o + (int64_t)g.nx * plane]
                                       : f4(ghost[(2 * g.ny + g.nx + ix) * N + jx]);
                else
                    hy = iy > 0 ? own[o - (int64_t)g.nx * plane] : f4(ghost[(2 * g.ny + ix) * N + jx]);
                dst[o] = upwind4(own[o], hx, hy, SX ? fabsf(scu[jx]) * fx : fabsf(scu[jx]), ay);
            }
        }
    }
}

// Eqs. densita..sforzi from float sums (see finalize_moments).
static __device__ __noinline__ void finalize_moments_f(const float *m, float e, double *o)
{
    const float rho = m[0], n = 1.f + e * rho;
    const float u[3] = {m[1] / n, m[2] / n, m[3] / n};
    o[0] = rho;
    o[1] = u[0];
    o[2] = u[1];
    o[3] = u[2];
    o[4] = ((2.f / 3.f) * (m[4] + m[5] + m[6]) - rho) / n -
           (2.f * e / 3.f) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const int pa[6] = {0, 1, 2, 0, 0, 1}, pb[6] = {0, 1, 2, 1, 2, 2};
    for (int k = 0; k < 6; ++k) o[5 + k] = 2.f * m[4 + k] - 2.f * e * n * u[pa[k]] * u[pb[k]];
}

// Per-instance shared tables of the FP32 cell kernel (N entries each).
__device__ __forceinline__ void cell4_setup(const Geo &g, const Cell4Smem &S)
{
    const int N = g.nv, T = blockDim.x, t = threadIdx.x;
    for (int i = t; i < N; i += T) {
        const double v = g.axv[i], A = g.axA[i];
        S.conv[i] = make_float4((float)A, (float)v, (float)(v * v), 0.f);
        S.gram[i] = make_float4((float)v, (float)(v * v), (float)(v * v * v), (float)(v * v * v * v));
        S.fin[i] = make_float4((float)(1.0 / A), 0.f, (float)A, (float)(A * v));
        S.Av2[i] = (float)(A * v * v);
        S.cu[i] = (float)(v * g.dt / g.dx);
        S.v[i] = (float)v;
        S.A[i] = (float)A;
        S.IA[i] = (float)(1.0 / A);
        S.rot[i] = i % (N / 4);
    }
    __syncthreads();
    for (int i = t; i < N / 4; i += T) {
        S.vzq[i] = make_float4(S.v[4 * i], S.v[4 * i + 1], S.v[4 * i + 2], S.v[4 * i + 3]);
        S.Azq[i] = make_float4(S.A[4 * i], S.A[4 * i + 1], S.A[4 * i + 2], S.A[4 * i + 3]);
        S.IAzq[i] = make_float4(S.IA[4 * i], S.IA[4 * i + 1], S.IA[4 * i + 2], S.IA[4 * i + 3]);
    }
    __syncthreads();
}

// One cell c of instance g: streaming into the slab (FUSED) or a copy of
// h~, the Monte Carlo gather and scatter, the correction and the write-back.
// Called by every thread of the CTA with the tables of g in place.
template <bool FUSED>
__device__ __forceinline__ void cell4_cell(const Geo &g, const Map4 &m, int c,
                                           const float *__restrict__ hin,
                                           const float *__restrict__ ghost,
                                           const PlanA<float, uint16_t> *__restrict__ pa,
                                           const uint32_t *__restrict__ ent,
                                           const int *__restrict__ meta, float *__restrict__ hout,
                                           double *__restrict__ mom, const Cell4Smem &S,
                                           int &fallback, long long *__restrict__ clk, int ncell)
{
    const int N = g.nv, nvt = g.nvt, T = blockDim.x, t = threadIdx.x;
    auto stamp = [&](int ph) {
        if (clk && blockIdx.x == 0 && t == 0 && ncell < kClkCells)
            clk[ncell * kClkPhases + ph] = clock64();
    };
    const float eps = g.epsf;
    float *totf = reinterpret_cast<float *>(S.tot);
    // Quad of this thread.
    const int Q = m.Q, nq = N / 4;
    const int q = t % Q, kchunk = t / Q;
    const bool active = kchunk < m.K;
    const int jy = q / nq, jz0 = 4 * (q % nq);
    const int jx0 = active ? kchunk * m.J : 0, jx1 = active ? jx0 + m.J : 0;
    (void)jz0;
    // Per-node constants of the quad (v_z, A_y A_z, 1/(A_y A_z), v_y^2 + v_z^2)
    // are re-read from shared tables inside each pass rather than kept live
    // across the whole cell: registers are the binding limit at 1024 threads.
#define QUAD_CONSTS                                                                  \
    const float vy = S.v[jy];                                                        \
    float vz[4], Ayz[4], IAyz[4], qq[4];                                             \
    {                                                                                \
        const float4 z4 = S.vzq[qz], a4 = S.Azq[qz], i4 = S.IAzq[qz];                \
        const float ay_ = S.A[jy], iay_ = S.IA[jy];                                  \
        vz[0] = z4.x; vz[1] = z4.y; vz[2] = z4.z; vz[3] = z4.w;                      \
        Ayz[0] = ay_ * a4.x; Ayz[1] = ay_ * a4.y; Ayz[2] = ay_ * a4.z; Ayz[3] = ay_ * a4.w; \
        IAyz[0] = iay_ * i4.x; IAyz[1] = iay_ * i4.y; IAyz[2] = iay_ * i4.z; IAyz[3] = iay_ * i4.w; \
        for (int i_ = 0; i_ < 4; ++i_) qq[i_] = vy * vy + vz[i_] * vz[i_];          \
    }                                                                                \
    (void)IAyz; (void)Ayz; (void)qq; (void)vz
    const float ry = g.ryf;
    const int half = N / 2;
    const int Q4 = Q;   // float4 stride of one jx-plane
    // Shared-memory position of this thread's quad in plane jx: quads of a row
    // are rotated by jx so that the jz-concentrated sample gathers spread over
    // all banks (the plan's node indices use the same order).
    const int qz = q % nq, rowq = jy * nq;
    auto phys = [&](int jx) {
        int r = qz + S.rot[jx];
        r -= r >= nq ? nq : 0;
        return jx * Q4 + rowq + r;
    };
    const int ix = c % g.nx, iy = c / g.nx;
    const float4 *own4 = reinterpret_cast<const float4 *>(hin + (int64_t)c * nvt);
    stamp(0);

    // ---- slab <- h~ ------------------------------------------------------
    if (active) {
        if (FUSED) {
            // Courant factors of this cell (its own widths on stretched grids).
            const float fx = g.sx ? (float)g.sx[ix] : 1.f, fy = g.sy ? (float)g.sy[iy] : ry;
            const float cuy = S.cu[jy] * fy, ay = fabsf(cuy);
            const int64_t plane = (int64_t)nvt / 4;
            if (ix > 0 && ix < g.nx - 1 && iy > 0 && iy < g.ny - 1) {
                // Interior cell: all upwind sources are neighbour slabs.
                const float4 *ys = cuy > 0.f ? own4 - (int64_t)g.nx * plane
                                             : own4 + (int64_t)g.nx * plane;
                const float4 *xr = own4 + plane, *xl = own4 - plane;
                const int e = min(jx1, half), b = max(jx0, half);
                if (!g.sx) {
#pragma unroll 4
                    for (int jx = jx0; jx < e; ++jx) {
                        const int o = jx * Q4 + q;
                        const float4 h0 = own4[o], hx = xr[o], hy = ys[o];
                        S.slab4[phys(jx)] = upwind4(h0, hx, hy, fabsf(S.cu[jx]), ay);
                    }
#pragma unroll 4
                    for (int jx = b; jx < jx1; ++jx) {
                        const int o = jx * Q4 + q;
                        const float4 h0 = own4[o], hx = xl[o], hy = ys[o];
                        S.slab4[phys(jx)] = upwind4(h0, hx, hy, fabsf(S.cu[jx]), ay);
                    }
                } else {
                    for (int jx = jx0; jx < e; ++jx) {
                        const int o = jx * Q4 + q;
                        const float4 h0 = own4[o], hx = xr[o], hy = ys[o];
                        S.slab4[phys(jx)] = upwind4(h0, hx, hy, fabsf(S.cu[jx]) * fx, ay);
                    }
                    for (int jx = b; jx < jx1; ++jx) {
                        const int o = jx * Q4 + q;
                        const float4 h0 = own4[o], hx = xl[o], hy = ys[o];
                        S.slab4[phys(jx)] = upwind4(h0, hx, hy, fabsf(S.cu[jx]) * fx, ay);
                    }
                }
            } else {
                const float4 *ys = nullptr;
                const float *yg = nullptr;
                if (cuy > 0.f) {
                    if (iy > 0) ys = own4 - (int64_t)g.nx * plane;
                    else yg = ghost + (2 * g.ny + ix) * N;
                } else {
                    if (iy < g.ny - 1) ys = own4 + (int64_t)g.nx * plane;
                    else yg = ghost + (2 * g.ny + g.nx + ix) * N;
                }
                for (int jx = jx0; jx < jx1; ++jx) {
                    const int o = jx * Q4 + q;
                    const float4 h0 = own4[o];
                    float4 hx;
                    if (jx < half)   // v_x < 0: right neighbour or right-wall ghost
                        hx = ix < g.nx - 1 ? own4[plane + o] : f4(ghost[(g.ny + iy) * N + jy]);
                    else             // v_x > 0: left neighbour or left-wall ghost
                        hx = ix > 0 ? own4[o - plane] : f4(ghost[iy * N + jy]);
                    const float4 hy = ys ? ys[o] : f4(yg[jx]);
                    S.slab4[phys(jx)] = upwind4(h0, hx, hy, fabsf(S.cu[jx]) * fx, ay);
                }
            }
        } else {
#pragma unroll 4
            for (int jx = jx0; jx < jx1; ++jx) S.slab4[phys(jx)] = own4[jx * Q4 + q];
        }
    }
    __syncthreads();

    stamp(1);
    // ---- phase A: g_l W_l on h~ (Jacobi) into shared memory ---------------
    {
        const float *slab = reinterpret_cast<const float *>(S.slab4);
        int l = t;
        for (; l + 15 * T < g.nt; l += 16 * T) {
            PlanA<float, uint16_t> rec[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) rec[u] = pa[l + u * T];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const int a = rec[u].a(), b = rec[u].b();
                const float ha = a >= 0 ? slab[a] : 0.f;
                const float hb = b >= 0 ? slab[b] : 0.f;
                S.gw[l + u * T] = (ha + hb + eps * ha * hb) * rec[u].W;
            }
        }
        for (; l < g.nt; l += T) {
            const PlanA<float, uint16_t> r = pa[l];
            const int a = r.a(), b = r.b();
            const float ha = a >= 0 ? slab[a] : 0.f;
            const float hb = b >= 0 ? slab[b] : 0.f;
            S.gw[l] = (ha + hb + eps * ha * hb) * r.W;
        }
    }
    __syncthreads();

    stamp(2);
    // ---- N = w h~ in place, with the invariants of h~ ----------------------
    float p0 = 0.f, p1 = 0.f, p3 = 0.f, p4 = 0.f;
    if (active) {
        QUAD_CONSTS;
#pragma unroll 4
        for (int jx = jx0; jx < jx1; ++jx) {
            const int o = phys(jx);
            float4 h = S.slab4[o];
            const float4 cv = S.conv[jx];        // {A, v, v^2, -}
            float n0 = h.x * (cv.x * Ayz[0]), n1 = h.y * (cv.x * Ayz[1]);
            float n2 = h.z * (cv.x * Ayz[2]), n3 = h.w * (cv.x * Ayz[3]);
            S.slab4[o] = make_float4(n0, n1, n2, n3);
            const float sn = (n0 + n1) + (n2 + n3);
            p0 += sn;
            p1 += sn * cv.y;
            p3 += n0 * vz[0] + n1 * vz[1] + n2 * vz[2] + n3 * vz[3];
            p4 += n0 * (cv.z + qq[0]) + n1 * (cv.z + qq[1]) + n2 * (cv.z + qq[2]) +
                  n3 * (cv.z + qq[3]);
        }
    }
    __syncthreads();

    stamp(3);
    // ---- phase B: gains and losses (Eq. monteCarloInt) --------------------
    // Each thread walks its run of the destination-sorted list, sums the
    // terms of one node in a register and adds the sum with one atomic.
    {
        float *slabw = reinterpret_cast<float *>(S.slab4);
        const int E = meta[0], C = meta[1];
        const int base = t * C, n = max(0, min(C, E - base));
        // Only the first and the last node of a run can be shared with the
        // neighbouring runs; they are added atomically, the others plainly.
        int cur = -1;
        bool first = true;
        float acc = 0.f;
        auto flush = [&](bool shared) {
            if (cur >= 0 && acc != 0.f) {
                if (shared) atomicAdd(slabw + cur, acc);
                else slabw[cur] += acc;
            }
        };
        auto term = [&](uint32_t w, float r) {
            const int dest = (int)(w >> 16);
            if (dest != cur) {
                flush(first);
                first = cur < 0;
                cur = dest;
                acc = 0.f;
            }
            acc += (w & 0x8000u) ? -r : r;
        };
        int i = 0;
        for (; i + 7 < n; i += 8) {
            uint32_t w[8];
            float r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = ent[(int64_t)(i + u) * T + t];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = S.gw[w[u] & 0x7FFFu];   // before any flush
#pragma unroll
            for (int u = 0; u < 8; ++u) term(w[u], r[u]);
        }
        for (; i < n; ++i) {
            const uint32_t w = ent[(int64_t)i * T + t];
            term(w, S.gw[w & 0x7FFFu]);
        }
        flush(true);
    }
    __syncthreads();

    stamp(4);
    // ---- moments of N_c for the correction (post pass) --------------------
    float acc[19];
    {
        QUAD_CONSTS;
        float s[4][5];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 5; ++k) s[i][k] = 0.f;
        if (active) {
#pragma unroll 2
            for (int jx = jx0; jx < jx1; ++jx) {
                float4 n = S.slab4[phys(jx)];
                const float4 gv = S.gram[jx];   // v, v^2, v^3, v^4
                const float nn[4] = {n.x, n.y, n.z, n.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    s[i][0] += nn[i];
                    s[i][1] += nn[i] * gv.x;
                    s[i][2] += nn[i] * gv.y;
                    s[i][3] += nn[i] * gv.z;
                    s[i][4] += nn[i] * gv.w;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 19; ++k) acc[k] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float z = vz[i], qi = qq[i];
            const float s0 = s[i][0], s1 = s[i][1], s2 = s[i][2], s3 = s[i][3], s4 = s[i][4];
            acc[0] += s0;
            acc[1] += s1;
            acc[2] += vy * s0;
            acc[3] += z * s0;
            acc[4] += s2;
            acc[5] += vy * vy * s0;
            acc[6] += z * z * s0;
            acc[7] += vy * s1;
            acc[8] += z * s1;
            acc[9] += vy * z * s0;
            acc[10] += s3 + qi * s1;
            acc[11] += vy * (s2 + qi * s0);
            acc[12] += z * (s2 + qi * s0);
            acc[13] += s4 + 2.f * qi * s2 + qi * qi * s0;
        }
        // The thread's share of the increment sums D (post minus pre over
        // its own nodes, so only thread-sized partial sums cancel).
        acc[14] = acc[0] - p0;
        acc[15] = acc[1] - p1;
        acc[16] = acc[2] - vy * p0;
        acc[17] = acc[3] - p3;
        acc[18] = (acc[4] + acc[5] + acc[6]) - p4;
    }
    block_reduce4<19>(acc, S.red, totf);
    stamp(5);

    // ---- correction solve (warp 0, which shares the residual of the
    // refinement) and per-cell tables --------------------------------------
    float *muf = reinterpret_cast<float *>(S.mu);
    if (t < 32) {
        float mu5[5];
        const bool ok = correction_spd(g, totf, mu5, t);
        if (t == 0) {
            if (ok) {
                for (int a = 0; a < 5; ++a) muf[a] = mu5[a];
            } else {
                double m8[5], Pd[19];
                for (int a = 0; a < 19; ++a) Pd[a] = (double)totf[a];
                int f2 = 0;
                correction_solve<float>(g, Pd, m8, &f2);
                ++fallback;
                for (int a = 0; a < 5; ++a) muf[a] = (float)m8[a];
            }
        }
    }
    __syncthreads();
    const float mu0 = muf[0], mux = muf[1], muy = muf[2], muz = muf[3], mu4 = muf[4];
    for (int i = t; i < N; i += T) S.fin[i].y = mux * S.v[i] + mu4 * S.v[i] * S.v[i];
    __syncthreads();
    stamp(6);

    // ---- corrected write-back and output moments ---------------------------
    float mo[10];
    {
        QUAD_CONSTS;
        float tt[4][3];
#pragma unroll
        for (int i = 0; i < 4; ++i) tt[i][0] = tt[i][1] = tt[i][2] = 0.f;
        float ct[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ct[i] = mu0 + muy * vy + muz * vz[i] + mu4 * qq[i];
        if (active) {
            float4 *dst4 = reinterpret_cast<float4 *>(hout + (int64_t)c * nvt);
#pragma unroll 2
            for (int jx = jx0; jx < jx1; ++jx) {
                const int o = jx * Q4 + q;
                float4 n = S.slab4[phys(jx)];
                const float4 fv = S.fin[jx];        // 1/A, cx, A, A v
                const float av2 = S.Av2[jx];
                const float nn[4] = {n.x, n.y, n.z, n.w};
                float hn[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float hc = nn[i] * (fv.x * IAyz[i]);
                    const float corr = ct[i] + fv.y;
                    hn[i] = hc + (1.f + eps * hc) * corr;
                    tt[i][0] += hn[i] * fv.z;
                    tt[i][1] += hn[i] * fv.w;
                    tt[i][2] += hn[i] * av2;
                }
                dst4[o] = make_float4(hn[0], hn[1], hn[2], hn[3]);
            }
        }
#pragma unroll
        for (int k = 0; k < 10; ++k) mo[k] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = Ayz[i], z = vz[i];
            const float t0 = a * tt[i][0], t1 = a * tt[i][1], t2 = a * tt[i][2];
            mo[0] += t0;
            mo[1] += t1;
            mo[2] += vy * t0;
            mo[3] += z * t0;
            mo[4] += t2;
            mo[5] += vy * vy * t0;
            mo[6] += z * z * t0;
            mo[7] += vy * t1;
            mo[8] += z * t1;
            mo[9] += vy * z * t0;
        }
    }
    stamp(7);
    block_reduce4<10>(mo, S.red, totf);
    if (t == 0 && mom) finalize_moments_f(totf, eps, mom + (int64_t)c * 11);
    __syncthreads();
    stamp(8);
}

template <bool FUSED, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
k_cell4(Geo g, Map4 m, const float *__restrict__ hin, const float *__restrict__ ghost,
        const PlanA<float, uint16_t> *__restrict__ pa, const uint32_t *__restrict__ ent,
        const int *__restrict__ meta, float *__restrict__ hout, double *__restrict__ mom,
        unsigned long long *__restrict__ stats, long long *__restrict__ clk,
        const int *__restrict__ gate = nullptr)
{
    if (gate && !gate[1]) return;
    extern __shared__ __align__(16) char smem_raw[];
    const Cell4Smem S = carve4(smem_raw, g.nv, g.nvt);
    cell4_setup(g, S);
    int fallback = 0, ncell = 0;
    for (int kc = blockIdx.x; kc < g.nr; kc += gridDim.x, ++ncell)
        cell4_cell<FUSED>(g, m, cell_of(g, kc), hin, ghost, pa, ent, meta, hout, mom, S,
                          fallback, clk, ncell);
    if (fallback && stats) atomicAdd(stats + 3, (unsigned long long)fallback);
}

}  // namespace bzk
