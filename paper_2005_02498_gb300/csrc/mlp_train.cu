// mlp_train.cu -- a minibatch of surrogate training on the tensor cores in two
// launches (the network and its layouts: mlp.cu).
//
// At a minibatch of 512 rows every GEMM is about 0.3 us of MMA, so a step is a
// chain of latencies: seven dependent layers (four forward, three backward)
// and the update.  As separate launches (7 GEMMs, 4 weight-gradient GEMMs, 19
// small kernels) a step took 255 us.
//
//   mlp_fb_kernel: the whole chain.  A cluster of eight CTAs owns 128 rows; each CTA
//   owns 32 of the 256 columns of every layer and keeps GELU'(Z) of its tile in
//   registers from the forward to the backward pass.  A layer's columns are written into
//   the operand buffers of all eight CTAs' shared memory, and a barrier of the cluster
//   is the hand-over; what only the weight gradients need goes to global memory
//   (transposed) while the others arrive, the next layer's weights are loaded while the
//   epilogue runs.
//   mlp_dw_kernel: every weight gradient dW = dZ^T H at once, 42 CTAs of 128 x 32
//   outputs over all rows, with Adam and the BF16 copies in the epilogue; the bias
//   gradients (row sums of dZ^T) in 98 more.
// What bounds it: latency.  At 512 rows a minibatch is 32 CTAs in the first launch (27 us:
// seven dependent products, each with a hand-over of some 5000 cycles) and 140 in the
// second (18 us).  Two epochs of 8192 rows in minibatches of 512 take 2.22 ms (57 us a
// minibatch with the host's shuffle, and copies of parameters and data) where one launch per
// product, transposition, reduction and update took 8.18 ms, and four CTAs of 64 columns
// that exchanged their activations through L2 2.65 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "mlp_train.cuh"
#include "tc_gemm.cuh"

namespace ptadd {

namespace {

constexpr int NIN = 30, NOUT = 6, NH = 256;
constexpr int FB_CL = 8;              // CTAs of a cluster
constexpr int FB_N = NH / FB_CL;      // columns of a layer per CTA
constexpr int FB_C = 8;               // columns per thread
constexpr int FB_T = 128 * FB_N / FB_C;  // threads: 4 TMEM lane groups x FB_N / FB_C slices
constexpr int A_CHUNK = 128 * 64 * 2; // one K-chunk of 64 of the A operand
constexpr int FB_A = 4 * A_CHUNK;     // A: 128 rows x K 256
constexpr int FB_B = 4 * FB_N * 64 * 2;
constexpr int FB_SMEM = 2 * FB_A + FB_B;
constexpr int DW_T = 256, DW_N = 32, DW_KC = 8;  // threads, columns per CTA, K-chunks of 64 in shared memory
constexpr int DW_B_CHUNK = DW_N * 64 * 2;
constexpr int DW_SMEM = DW_KC * (A_CHUNK + DW_B_CHUNK);

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// generic-proxy writes to any CTA's shared memory before the tensor core's reads
__device__ __forceinline__ void fence_async_cluster() { asm volatile("fence.proxy.async.shared::cluster;" ::: "memory"); }

// K columns k0 .. k0 + 64 nchunk - 1 of rows row0 .. row0 + R - 1 of a K-contiguous matrix
// into nchunk consecutive chunks in the canonical layout (tc_gemm.cuh); zeros beyond row_lim and K.
template <int R, int T>
__device__ __forceinline__ void load_operand(uint32_t dst, const __nv_bfloat16* src, int64_t ld, int64_t row0,
                                             int64_t row_lim, int64_t k0, int64_t K, int nchunk)
{
    for (int v = threadIdx.x; v < nchunk * R * 8; v += T) {
        const int c = v / (R * 8), u = v - c * (R * 8);
        const int r = (u >> 6) * 8 + (u & 7), kk = (u >> 3) & 7;
        const int64_t gr = row0 + r, gk = k0 + 64 * c + 8 * kk;
        const bool in = gr < row_lim && gk < K;
        const __nv_bfloat16* p = in ? src + gr * ld + gk : src;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + c * (R * 128) + (r >> 3) * 1024 +
                                                                          kk * 128 + (r & 7) * 16),
                     "l"(__cvta_generic_to_global(p)), "r"(in ? 16u : 0u)
                     : "memory");
    }
}

// D (+)= A B^T over `steps` K-steps of 16 from the chunks at a0 and b0 (R_B rows of B).
template <int R_B>
__device__ __forceinline__ void issue_mma(uint32_t tmem, uint32_t a0, uint32_t b0, int steps, uint32_t idesc, bool add)
{
    for (int s = 0; s < steps; ++s) {
        const uint32_t c = s >> 2, o = (s & 3) * 256;
        tc_mma_f16(tmem, smem_desc(a0 + c * A_CHUNK + o, 128, 1024), smem_desc(b0 + c * (R_B * 128) + o, 128, 1024),
                   idesc, (add || s > 0) ? 1u : 0u);
    }
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// FB_C values of a tile's row lr, columns c .. c + FB_C - 1, in BF16: into the A operand at
// shared-memory address a of the CTAs 0 .. peers - 1 of the cluster
__device__ __forceinline__ void share8(const float h[FB_C], uint32_t a, int lr, int c, int peers)
{
    const uint32_t at = a + (uint32_t)((c >> 6) * A_CHUNK + (lr >> 3) * 1024 + ((c >> 3) & 7) * 128 + (lr & 7) * 16);
    const uint32_t w0 = pack2(h[0], h[1]), w1 = pack2(h[2], h[3]), w2 = pack2(h[4], h[5]), w3 = pack2(h[6], h[7]);
#pragma unroll
    for (int p = 0; p < FB_CL; ++p) {
        if (p >= peers) break;
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(at), "r"(p));
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w0), "r"(w1), "r"(w2), "r"(w3)
                     : "memory");
    }
    fence_async_cluster();
}
// ... and transposed [. x rows] for the weight gradients
__device__ __forceinline__ void store_t8(const float h[FB_C], __nv_bfloat16* tr, int64_t rows, int64_t r, int c)
{
#pragma unroll
    for (int i = 0; i < FB_C; ++i) tr[(int64_t)(c + i) * rows + r] = __float2bfloat16_rn(h[i]);
}
// 8 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float v[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])::"memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__global__ void __cluster_dims__(1, FB_CL, 1) __launch_bounds__(FB_T, 1) mlp_fb_kernel(TrainArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float red[4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t row0 = (int64_t)blockIdx.x * 128;
    const int y = blockIdx.y, n0 = y * FB_N;
    const uint32_t uA = smem_u32(smem), uB = uA + 2 * FB_A, mb = smem_u32(&mbar);
    const int lr = 32 * (warp & 3) + lane;  // this thread's row of the tile
    const int c0 = FB_C * (warp >> 2);      // and first column of its slice
    const int64_t r = row0 + lr;
    const bool live = r < g.rows;
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_base), FB_N);
        tmem_relinquish();
    }
    if (tid == 0) mbar_init(mb, 1);
    cluster_arrive();  // (waited for before the first write into another CTA: it has started by then)
    // layer 1: its weights, and the inputs straight from the samples
    load_operand<FB_N, FB_T>(uB, g.Wb[0], din_p(0), n0, NH, 0, din_p(0), 1);
    cp_commit();
    for (int e = tid; e < 128 * 4; e += FB_T) {
        const int xr = e >> 2, part = e & 3;
        const int64_t gr = row0 + xr;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.0f;
        if (gr < g.n) {
            const float* p = g.xn + (g.idx ? (int64_t)g.idx[gr] : gr) * NIN + 8 * part;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (8 * part + i < NIN) v[i] = p[i];
        }
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = pack2(v[2 * i], v[2 * i + 1]);
        *reinterpret_cast<uint4*>(smem + (xr >> 3) * 1024 + part * 128 + (xr & 7) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        if (y == 1 && gr < g.rows)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
                g.Xt[(int64_t)(8 * part + 2 * i) * g.rows + gr] = h.x;
                g.Xt[(int64_t)(8 * part + 2 * i + 1) * g.rows + gr] = h.y;
            }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base, trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
    uint32_t phase = 0;
    bool ok = true;
    // the operands have been issued: wait for them, multiply, wait for the product.  A wait
    // that gives up leaves the rest of the tile's products out; every barrier is still met.
    auto multiply = [&](uint32_t ua, int steps, int N) {
        cp_wait_all();
        fence_async_cluster();  // this thread's copies, and what its barrier wait has made visible
        tc_fence_before();
        __syncthreads();
        if (tid == 0 && ok) {
            tc_fence_after();
            issue_mma<FB_N>(tmem, ua, uB, steps, idesc_bf16_f32(128, N), false);
            tc_commit(mb);
        }
        bool w = true;
        if (ok) w = mbar_wait_bounded(mb, phase, MBAR_WAIT_LIMIT);
        phase ^= 1u;
        ok = __syncthreads_and(ok && w);
        tc_fence_after();
    };
    // The A operand alternates between two buffers (layer l reads buffer l mod 2): a CTA writes
    // its columns of the next operand while a slower one still multiplies from this one, and
    // a buffer's last readers have passed a barrier of the cluster before it is written again.
    float dg[3][FB_C];  // GELU'(Z) of this thread's values
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        multiply(uA + (l & 1) * FB_A, l == 0 ? 2 : 16, FB_N);
        // the next layer's weights, while the epilogue runs
        if (l < 2)
            load_operand<FB_N, FB_T>(uB, g.Wb[l + 1], NH, n0, NH, 0, NH, 4);
        else if (y == 0)
            load_operand<FB_N, FB_T>(uB, g.Wb[3], NH, 0, dout_p(3), 0, NH, 4);
        cp_commit();
        float z[FB_C], h[FB_C], e[FB_C];
        tmem_ld8(trow, z);
#pragma unroll
        for (int i = 0; i < FB_C; ++i) {
            z[i] += g.b[l][n0 + c0 + i];
            e[i] = 1.0f + erff(z[i] * 0.70710678118654752f);
            h[i] = 0.5f * z[i] * e[i];
        }
        if (l == 0) cluster_wait();
        share8(h, uA + ((l + 1) & 1) * FB_A, lr, n0 + c0, l < 2 ? FB_CL : 1);  // (layer 4 is the first CTA's)
        tc_fence_before();
        cluster_arrive();
        // what only the backward pass and the weight gradients read, while the others arrive
        if (live) store_t8(h, g.Ht[l], g.rows, r, n0 + c0);
#pragma unroll
        for (int i = 0; i < FB_C; ++i)
            dg[l][i] = 0.5f * e[i] + z[i] * expf(-0.5f * z[i] * z[i]) * 0.39894228040143268f;
        cluster_wait();
    }
    // layer 4 (one CTA of the cluster), the loss and its gradient
    if (y == 0) {
        multiply(uA + FB_A, 16, dout_p(3));
        load_operand<FB_N, FB_T>(uB, g.Wt[3], dout_p(3), n0, NH, 0, dout_p(3), 1);
        cp_commit();
        if (c0 < dout_p(3)) {
            float v[FB_C], d[FB_C], loss = 0.0f;
            tmem_ld8(trow, v);
            const float scale = 1.0f / ((float)g.n * NOUT);
            const bool in = r < g.n;
            const float* t = g.yn + (in ? (g.idx ? (int64_t)g.idx[r] : r) : 0) * NOUT;
#pragma unroll
            for (int i = 0; i < FB_C; ++i) {
                d[i] = 0.0f;
                if (in && c0 + i < NOUT) {
                    const float e = v[i] + g.b[3][c0 + i] - t[c0 + i];
                    loss += e * e * scale;
                    d[i] = 2.0f * e * scale;
                }
            }
            share8(d, uA, lr, c0, FB_CL);
            if (live) store_t8(d, g.dYt, g.rows, r, c0);
            if (c0 == 0) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
                if (lane == 0) red[warp] = loss;
            }
        }
        __syncthreads();
        if (tid == 0) g.loss_part[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
    } else {
        load_operand<FB_N, FB_T>(uB, g.Wt[3], dout_p(3), n0, NH, 0, dout_p(3), 1);
        cp_commit();
    }
    tc_fence_before();
    cluster_arrive();
    cluster_wait();
    // backward: dZ_l = (dZ_{l+1} W_{l+1}) GELU'(Z_l)
#pragma unroll
    for (int l = 2; l >= 0; --l) {
        multiply(uA + (l & 1) * FB_A, l == 2 ? 1 : 16, FB_N);
        if (l > 0) {
            load_operand<FB_N, FB_T>(uB, g.Wt[l], NH, n0, NH, 0, NH, 4);
            cp_commit();
        }
        float v[FB_C];
        tmem_ld8(trow, v);
#pragma unroll
        for (int i = 0; i < FB_C; ++i) v[i] *= dg[l][i];
        if (l > 0) {
            share8(v, uA + ((l - 1) & 1) * FB_A, lr, n0 + c0, FB_CL);
            tc_fence_before();
            cluster_arrive();
        }
        if (live) store_t8(v, g.dZt[l], g.rows, r, n0 + c0);
        if (l > 0) cluster_wait();
    }
    if (!ok && tid == 0) {
        atomicExch(g.err, 1);
        // a last bounded chance for the tensor core before its memory is freed
        mbar_wait_bounded(mb, 0u, MBAR_WAIT_LIMIT);
        mbar_wait_bounded(mb, 1u, MBAR_WAIT_LIMIT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, FB_N);
}

__device__ __forceinline__ float adam_step(float p, float g, float& m, float& v, const TrainArgs& a)
{
    m = __fmaf_rn(1.0f - a.b1, g, __fmul_rn(a.b1, m));
    v = __fmaf_rn(__fmul_rn(1.0f - a.b2, g), g, __fmul_rn(a.b2, v));
    return p - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

constexpr int DW_TILES = 2 + 16 + 16 + 8;
constexpr int BIAS_ROWS = 256 + 256 + 256 + 16;

// Bias gradients: row sums of dZ^T, one warp per row, with the update.
__device__ __forceinline__ void bias_rows(const TrainArgs& g, int row)
{
    const int l = row < 768 ? row >> 8 : 3, o = row - 256 * l, lane = threadIdx.x & 31;
    const __nv_bfloat16* p = (l == 3 ? g.dYt : g.dZt[l]) + (int64_t)o * g.rows;
    float s = 0.0f;
#pragma unroll 8
    for (int64_t k = lane; k < g.rows; k += 32) s += __bfloat162float(p[k]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if (lane != 0) return;
    if (!g.adam) {
        g.gb[l][o] = s;
        return;
    }
    float m = g.mb[l][o], v = g.vb[l][o];
    g.b[l][o] = adam_step(g.b[l][o], s, m, v, g);
    g.mb[l][o] = m;
    g.vb[l][o] = v;
}

// CTA: one 128 x 32 tile of one layer's weight gradient (tile order: layer 1's 2, 16
// each of layers 2 and 3, layer 4's 8); the CTAs after them eight bias rows each.
__global__ void __launch_bounds__(DW_T, 1) mlp_dw_kernel(TrainArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int t = blockIdx.x, l = 0;
    if (t >= DW_TILES) {
        bias_rows(g, (t - DW_TILES) * (DW_T / 32) + warp);
        return;
    }
    if (t >= 2) {
        t -= 2;
        l = 1 + t / 16;
        t %= 16;
    }
    const int nt = din_p(l) / DW_N;  // column tiles
    const int m0 = 128 * (t / nt), n0 = DW_N * (t % nt);
    const __nv_bfloat16* A = l == 3 ? g.dYt : g.dZt[l];
    const __nv_bfloat16* B = l == 0 ? g.Xt : g.Ht[l - 1];
    const uint32_t uA = smem_u32(smem), uB = uA + DW_KC * A_CHUNK, mb = smem_u32(&mbar);
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_base), DW_N);
        tmem_relinquish();
    }
    if (tid == 0) mbar_init(mb, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    uint32_t phase = 0;
    bool ok = true;
    for (int64_t k0 = 0; k0 < g.rows && ok; k0 += 64 * DW_KC) {
        const int kn = (int)min((int64_t)64 * DW_KC, g.rows - k0), nc = (kn + 63) / 64;
        load_operand<128, DW_T>(uA, A, g.rows, m0, dout_p(l), k0, g.rows, nc);
        load_operand<DW_N, DW_T>(uB, B, g.rows, n0, din_p(l), k0, g.rows, nc);
        cp_commit();
        cp_wait_all();
        fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            issue_mma<DW_N>(tmem, uA, uB, kn / 16, idesc_bf16_f32(128, DW_N), k0 > 0);
            tc_commit(mb);
        }
        ok = mbar_wait_bounded(mb, phase, MBAR_WAIT_LIMIT);
        phase ^= 1u;
        ok = __syncthreads_and(ok);
    }
    tc_fence_after();
    if (ok) {
        const int o = m0 + 32 * (warp & 3) + lane, c = n0 + 16 * (warp >> 2);
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(16 * (warp >> 2)), v);
        if (o < dout_p(l)) {
            const int64_t at = (int64_t)o * din_p(l) + c;
            if (!g.adam) {
                float4* out = reinterpret_cast<float4*>(g.gW[l] + at);
#pragma unroll
                for (int i = 0; i < 4; ++i) out[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            } else {
                float4* pw = reinterpret_cast<float4*>(g.W[l] + at);
                float4* pm = reinterpret_cast<float4*>(g.mW[l] + at);
                float4* pv = reinterpret_cast<float4*>(g.vW[l] + at);
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float4 p = pw[i], m = pm[i], s = pv[i];
                    p.x = adam_step(p.x, v[4 * i], m.x, s.x, g);
                    p.y = adam_step(p.y, v[4 * i + 1], m.y, s.y, g);
                    p.z = adam_step(p.z, v[4 * i + 2], m.z, s.z, g);
                    p.w = adam_step(p.w, v[4 * i + 3], m.w, s.w, g);
                    pw[i] = p;
                    pm[i] = m;
                    pv[i] = s;
                    w[2 * i] = pack2(p.x, p.y);
                    w[2 * i + 1] = pack2(p.z, p.w);
                }
                uint4* wb = reinterpret_cast<uint4*>(g.Wb[l] + at);
                wb[0] = make_uint4(w[0], w[1], w[2], w[3]);
                wb[1] = make_uint4(w[4], w[5], w[6], w[7]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
                    g.Wt[l][(int64_t)(c + 2 * i) * dout_p(l) + o] = h.x;
                    g.Wt[l][(int64_t)(c + 2 * i + 1) * dout_p(l) + o] = h.y;
                }
            }
        }
    } else if (tid == 0) {
        atomicExch(g.err, 1);
        mbar_wait_bounded(mb, phase ^ 1u, MBAR_WAIT_LIMIT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, DW_N);
}

}  // namespace

cudaError_t launch_mlp_train(const TrainArgs& g, cudaStream_t s)
{
    static bool attr_set[64] = {};  // the attributes are per function and device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(mlp_fb_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(mlp_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    if (g.rows <= 0) return cudaSuccess;
    mlp_fb_kernel<<<dim3((unsigned)((g.rows + 127) / 128), FB_CL), FB_T, FB_SMEM, s>>>(g);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mlp_dw_kernel<<<DW_TILES + BIAS_ROWS / (DW_T / 32), DW_T, DW_SMEM, s>>>(g);
    return cudaGetLastError();
}

}  // namespace ptadd
