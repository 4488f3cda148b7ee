// step.cu -- the O(N) phases of a DD step (step.cuh).
//
// On this GPU a warp's FP64 instruction occupies its scheduler's FP64 unit for 64
// cycles (half a lane per cycle), so for the networks of a few hundred to a few
// thousand nodes, which do not fill the SMs, these phases cost their FP64
// instruction count in latency.  Hence one launch instead of four or five, the
// segment lengths read back from the source records, sums by halves across a warp
// (16 additions for 13 values instead of 65), and averages kept as running
// sums per group that are added up once per burst.  Beside the pair kernel a step of
// 512 segments (one-loop groups) took 45 us in five launches and takes 21 in one; of
// 1485 segments with the consistent mobility 505 us (one thread per loop walked
// its elimination: 460) and now 44.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "chain.cuh"
#include "pair_tile.cuh"
#include "step.cuh"

namespace ptadd {

namespace {

constexpr int NSUM = 13;

// Sums of 16 values over a warp: at each of four exchanges a lane keeps half of
// its values, so lane l ends with the total of value l >> 1.
__device__ __forceinline__ double warp_sum16(double v[16])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < h) {
                const double keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Consistent mobility (Eq. 2.1's weak form with linear shape functions, internal
// units, B = 1): sum_b M_ab v_b = P F_a on each ring, M_aa = (L_prev + L_next)/3,
// M_a,a+-1 = L/6 of the segment between them, v = 0 at held nodes (pinned, or
// both segments of zero length).  Row a is kept as v_a + p v_a-s + q v_a+s = d with
// s = 1, 2, 4, ... (cyclic reduction of every row at once, neighbours taken
// around the ring).  |p| + |q| <= 1/2 at the start and is at most squared by each
// step, 2^-64 after the sixth: beyond FP64's rounding, and v = d.  Rings of any
// length and chains between held nodes need no case of their own.
__device__ __forceinline__ bool step_held(const StepArgs& a, int64_t i, double Lp, double Ln)
{
    return a.pinned[i] != 0 || !(Lp + Ln > 0.0);
}
__device__ __forceinline__ double seg_length(const StepArgs& a, int64_t i) { return a.src[SRC_STRIDE * i + 3]; }

__device__ __forceinline__ void reduce_row(const StepArgs& a, int64_t i, int k)
{
    const double* x = a.scr + (k & 1) * 5 * a.n;
    const int lp = a.loop_of[i];
    const int64_t b = a.loop_off[lp], m = a.loop_off[lp + 1] - b;
    const int64_t s = (int64_t)(1 << k) % m;
    int64_t lo = i - s, hi = i + s;
    if (lo < b) lo += m;
    if (hi >= b + m) hi -= m;
    const int64_t n = a.n;
    const double p = x[i], q = x[n + i], p0 = x[lo], q0 = x[n + lo], p1 = x[hi], q1 = x[n + hi];
    const double r = 1.0 / fma(-q, p1, fma(-p, q0, 1.0));
    double d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double* e = x + (2 + c) * n;
        d[c] = fma(-q, e[hi], fma(-p, e[lo], e[i])) * r;
    }
    if (k == 5) {
#pragma unroll
        for (int c = 0; c < 3; ++c) a.vel[c * n + i] = d[c];
        return;
    }
    double* y = a.scr + ((k & 1) ^ 1) * 5 * n;
    y[i] = -p * p0 * r;
    y[n + i] = -q * q1 * r;
#pragma unroll
    for (int c = 0; c < 3; ++c) y[(2 + c) * n + i] = d[c];
}

// One reduction step of the consistent system over all nodes (rings too long for a block).
__global__ void step_reduce_kernel(StepArgs a, int k)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < a.n) reduce_row(a, i, k);
}

// Where the parts of node i's realisation lie: its nodes' number, i within it, the chunks.
struct PartView {
    const double* fp;
    int64_t nr, off;
    int chunks;
};
__device__ __forceinline__ PartView part_view(const StepArgs& a, int64_t i)
{
    if (!a.real_of) return PartView{a.fpart, a.n, 0, a.chunks};
    const int r = a.real_of[i];
    const int64_t o = a.node_off[r];
    return PartView{a.fpart + a.fp_base[r], a.node_off[r + 1] - o, o, a.chunks_of[r]};
}
// Adds the chunks row, row + rows, ... of node i (previous node p on its loop) to F.
__device__ __forceinline__ void sum_parts(const StepArgs& a, int64_t i, int64_t p, int row, int rows, double F[3])
{
    const PartView w = part_view(a, i);
    const int64_t li = i - w.off, lq = p - w.off;
#pragma unroll 4
    for (int ch = row; ch < w.chunks; ch += rows) {
        const double* f = w.fp + (int64_t)ch * 6 * w.nr;
#pragma unroll
        for (int e = 0; e < 3; ++e) F[e] += f[e * w.nr + li] + f[(3 + e) * w.nr + lq];
    }
}

constexpr int NF_ROWS = 8;

// Block: 32 nodes x NF_ROWS rows of chunks; the rows are added in order.
__global__ void __launch_bounds__(32 * NF_ROWS) node_force_kernel(StepArgs a, double* __restrict__ force)
{
    __shared__ double red[NF_ROWS][3][32];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + lane;
    const bool live = i < a.n && !(a.real_of && a.pinned[i]);
    double F[3] = {0.0, 0.0, 0.0};
    if (live) sum_parts(a, i, a.prv[i], row, NF_ROWS, F);
#pragma unroll
    for (int e = 0; e < 3; ++e) red[row][e][lane] = F[e];
    __syncthreads();
    if (row != 0 || i >= a.n) return;
#pragma unroll
    for (int y = 1; y < NF_ROWS; ++y)
#pragma unroll
        for (int e = 0; e < 3; ++e) F[e] += red[y][e][lane];
#pragma unroll
    for (int e = 0; e < 3; ++e) force[e * a.n + i] = F[e];
}

// Block: one group, 32 nodes x ROWS at a time.
template <int ROWS>
__global__ void __launch_bounds__(32 * ROWS) step_kernel(StepArgs a, int what)
{
    __shared__ double red[ROWS][3][33];
    const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
    chain_wait();
    // In the middle of a step the next kernel's few blocks may be set up beside these.  At its end the
    // next kernel is the pair stage, sized to fill the SMs once: set up around these blocks it
    // would be spread unevenly (512 segments: 78 against 75 us a step), so it comes as they end.
    if (!(what & STEP_EULER)) chain_next();
    const int64_t lo = a.grp_off[blockIdx.x], hi = a.grp_off[blockIdx.x + 1], n = a.n;
    if (a.counter && blockIdx.x == 0 && tid == 0) *a.counter = 0u;
    if (what & STEP_NODE) {
        for (int64_t base = lo; base < hi; base += 32) {
            const int64_t i = base + lane;
            const bool live = i < hi && !a.pinned[i];
            const int64_t p = live ? a.prv[i] : 0;
            double F[3] = {0.0, 0.0, 0.0};
            if (live) sum_parts(a, i, p, row, ROWS, F);
#pragma unroll
            for (int e = 0; e < 3; ++e) red[row][e][lane] = F[e];
            __syncthreads();
            // rows in two levels, in a fixed order
            if (ROWS > 4 && row < 4)
                for (int y = row + 4; y < ROWS; y += 4)
#pragma unroll
                    for (int e = 0; e < 3; ++e) red[row][e][lane] += red[y][e][lane];
            if (ROWS > 4) __syncthreads();
            if (row == 0 && i < hi) {
                double v[3] = {0.0, 0.0, 0.0}, cp = 0.0, cq = 0.0;
                if (live) {
#pragma unroll
                    for (int e = 0; e < 3; ++e)
                        F[e] = (red[0][e][lane] + red[1][e][lane]) + (red[2][e][lane] + red[3][e][lane]);
                    const double Lp = seg_length(a, p), Ln = seg_length(a, i);
                    const int k = a.loop_of[i];
                    const double nn[3] = {a.loop_n[3 * k], a.loop_n[3 * k + 1], a.loop_n[3 * k + 2]};
                    const double nF = fma(nn[0], F[0], fma(nn[1], F[1], nn[2] * F[2]));
                    if (Lp + Ln > 0.0) {
                        double inv = 2.0 / (Lp + Ln);
                        if (what & STEP_CONSISTENT) {
                            inv *= 1.5;  // 1 / M_aa
                            const int64_t q = a.nxt[i], pp = a.prv[p];
                            cp = step_held(a, p, seg_length(a, pp), Lp) ? 0.0 : Lp * (1.0 / 6.0) * inv;
                            cq = step_held(a, q, Ln, seg_length(a, q)) ? 0.0 : Ln * (1.0 / 6.0) * inv;
                        }
#pragma unroll
                        for (int e = 0; e < 3; ++e) v[e] = fma(-nn[e], nF, F[e]) * inv;
                    }
                }
                if (what & STEP_CONSISTENT) {
                    a.scr[i] = cp;
                    a.scr[n + i] = cq;
#pragma unroll
                    for (int e = 0; e < 3; ++e) a.scr[(2 + e) * n + i] = v[e];
                } else {
#pragma unroll
                    for (int e = 0; e < 3; ++e) a.vel[e * n + i] = v[e];
                }
            }
            __syncthreads();
        }
    }
    if ((what & STEP_CONSISTENT) && !(what & STEP_ROWS))
        for (int k = 0; k < 6; ++k) {
            for (int64_t i = lo + tid; i < hi; i += 32 * ROWS) reduce_row(a, i, k);
            __syncthreads();
        }
    if (!(what & STEP_EULER)) return;

    double v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = 0.0;
    for (int64_t i = lo + tid; i < hi; i += 32 * ROWS) {
        const int64_t j = a.nxt[i];
        const int k = a.loop_of[i];
        double x1[3], x2[3], v1[3], D[3], vb[3];
        const double b[3] = {a.loop_b[3 * k], a.loop_b[3 * k + 1], a.loop_b[3 * k + 2]};
        const double L = seg_length(a, i);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            x1[e] = a.pos[e * n + i];
            x2[e] = a.pos[e * n + j];
            v1[e] = a.vel[e * n + i];
            const double v2 = a.vel[e * n + j];
            D[e] = x2[e] - x1[e];
            vb[e] = 0.5 * (v1[e] + v2);
            // explicit Euler (all nodes from the step-start state)
            x1[e] = __dadd_rn(x1[e], __dmul_rn(v1[e], a.dt));
            x2[e] = __dadd_rn(x2[e], __dmul_rn(v2, a.dt));
            a.pos_next[e * n + i] = x1[e];
            v[10 + e] = fma(L, vb[e], v[10 + e]);
        }
        if (!isfinite(x1[0]) || !isfinite(x1[1]) || !isfinite(x1[2])) atomicOr(a.flag, 1);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int f = (e + 1) % 3, g = (e + 2) % 3;
            const double c = fma(D[f], vb[g], -(D[g] * vb[f]));  // L t x vbar
#pragma unroll
            for (int m = 0; m < 3; ++m) v[3 * m + e] = fma(b[m], c, v[3 * m + e]);
        }
        v[9] += L;
        if (what & STEP_PREP) {
            const double* o = a.origin ? a.origin + 3 * a.real_of[i] : a.org;
            const double og[3] = {o[0], o[1], o[2]};
            seg_records(x1, x2, b, og, a.a2, a.src + (int64_t)SRC_STRIDE * i,
                        a.src32 ? a.src32 + (int64_t)SRC32_STRIDE * i : nullptr,
                        a.srcdf ? a.srcdf + (int64_t)SRCDF_STRIDE * i : nullptr);
        }
    }
    // warps that hold nodes: their sums, then those of the group in order
    const int nw = (int)min((int64_t)ROWS, (hi - lo + 31) / 32);
    double s = 0.0;
    if (row < nw) s = warp_sum16(v);
    double* out = a.part + 16 * (int64_t)blockIdx.x;
    if (nw > 1) {
        __syncthreads();
        if (row < nw && !(lane & 1)) red[row][0][lane >> 1] = s;
        __syncthreads();
        if (row == 0 && !(lane & 1))
            for (int y = 1; y < nw; ++y) s += red[y][0][lane >> 1];
    }
    if (row == 0 && !(lane & 1) && (lane >> 1) < NSUM) {
        out[lane >> 1] = fma(s, a.dt, out[lane >> 1]);
        if ((lane >> 1) == 9) out[13] = s;
    }
}

// Block: one realisation; thread (m, y): value m of the groups y, y + 16, ..., then the
// 16 partial sums in order.
__global__ void __launch_bounds__(256) step_finish_kernel(const int32_t* __restrict__ real_grp,
                                                          const double* __restrict__ part, int length_only,
                                                          double* __restrict__ acc)
{
    __shared__ double red[16][16];
    const int m = threadIdx.x & 15, y = threadIdx.x >> 4;
    const int g0 = real_grp[blockIdx.x], g1 = real_grp[blockIdx.x + 1];
    double s = 0.0;
    if (m <= NSUM)
        for (int g = g0 + y; g < g1; g += 16) s += part[16 * (int64_t)g + m];
    red[y][m] = s;
    __syncthreads();
    if (y != 0) return;
    for (int k = 1; k < 16; ++k) s += red[k][m];
    double* a = acc + 16 * (int64_t)blockIdx.x;
    if (length_only) {
        if (m == NSUM) a[11] = s;
    } else if (m < NSUM) {
        a[m < 10 ? m : m + 3] += s;
    }
}

}  // namespace

StepGroups step_groups(int64_t n_loops, const int64_t* loop_off, int32_t R, const int64_t* node_off)
{
    StepGroups g;
    for (int64_t k = 0; k < n_loops; ++k)
        if (loop_off[k + 1] - loop_off[k] > STEP_LOOP_MAX) g.whole = false;
    int64_t k = 0;
    for (int32_t r = 0; r < R; ++r) {
        g.real_grp.push_back((int32_t)g.off.size());
        const int64_t end = node_off[r + 1];
        if (!g.whole) {
            for (int64_t i = node_off[r]; i < end; i += 32) g.off.push_back((int32_t)i);
            continue;
        }
        while (k < n_loops && loop_off[k] < end) {
            const int64_t first = loop_off[k++];
            g.off.push_back((int32_t)first);
            while (k < n_loops && loop_off[k] < end && loop_off[k + 1] - first <= 32) ++k;
        }
    }
    g.real_grp.push_back((int32_t)g.off.size());
    g.off.push_back((int32_t)node_off[R]);
    return g;
}

cudaError_t launch_step(const StepArgs& a, int n_groups, bool whole, int max_chunks, int what, cudaStream_t st,
                        int64_t* launches, bool chained)
{
    if (a.n == 0) return cudaSuccess;
    auto go = [&](int w) {
        // 16 rows where at most one block per SM sums many chunks: its rows shorten the chain of
        // sums.  With more blocks than SMs, or few chunks, 4 rows: the others would
        // only take part in barriers.  us a step with 16 / 4 rows: 64 groups 134.8 / 137.8 (mixed), 459.6 / 466.8
        // (FP64); 128 groups equal; 192 groups 600.6 / 593.0, 3635 / 3625; 256 groups 971 / 966, 6244 / 6238; 16 groups of 2
        // chunks 74.7 / 74.2.
        *launches += 1;
        const bool tall = max_chunks > 16 && n_groups <= device_sms();
        if (chained)
            return tall ? launch_chained(step_kernel<16>, n_groups, 512, 0, st, a, w)
                        : launch_chained(step_kernel<4>, n_groups, 128, 0, st, a, w);
        if (tall)
            step_kernel<16><<<n_groups, 512, 0, st>>>(a, w);
        else
            step_kernel<4><<<n_groups, 128, 0, st>>>(a, w);
        return cudaGetLastError();
    };
    if (whole) return go(what);
    cudaError_t e = cudaSuccess;
    if (what & STEP_NODE) {
        e = go((what & (STEP_NODE | STEP_CONSISTENT)) | STEP_ROWS);
        if (e != cudaSuccess) return e;
        if (what & STEP_CONSISTENT)
            for (int k = 0; k < 6; ++k) {
                step_reduce_kernel<<<(unsigned)((a.n + 127) / 128), 128, 0, st>>>(a, k);
                *launches += 1;
                e = cudaGetLastError();
                if (e != cudaSuccess) return e;
            }
    }
    if (what & STEP_EULER) e = go(what & ~(STEP_NODE | STEP_CONSISTENT));
    return e;
}

cudaError_t launch_node_force(const StepArgs& a, double* force, cudaStream_t st)
{
    if (a.n == 0) return cudaSuccess;
    node_force_kernel<<<(unsigned)((a.n + 31) / 32), 32 * NF_ROWS, 0, st>>>(a, force);
    return cudaGetLastError();
}

cudaError_t launch_step_finish(int32_t R, const int32_t* real_grp, const double* part, bool length_only, double* acc,
                               cudaStream_t st)
{
    step_finish_kernel<<<R, 256, 0, st>>>(real_grp, part, length_only ? 1 : 0, acc);
    return cudaGetLastError();
}

}  // namespace ptadd
