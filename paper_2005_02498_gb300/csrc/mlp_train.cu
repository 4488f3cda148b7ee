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
//   registers from the forward to the backward pass.  A layer's columns are one
//   contiguous piece of the next layer's operand: written in the CTA's own shared
//   memory and sent to the other seven by bulk copies that complete on the receiver's
//   mbarrier.  What only the weight gradients need goes to global memory while the
//   pieces are on their way, transposed and already in the operand layout; the next layer's
//   weights are loaded while the epilogue runs.
//   mlp_dw_kernel: every weight gradient dW = dZ^T H at once, 42 CTAs of 128 x 32
//   outputs over all rows, operands by bulk copies, with Adam (parameters and moments
//   loaded while the operands arrive) and the BF16 copies in the epilogue; the bias
//   gradients (row sums of dZ^T) in 49 more.
// What bounds it: latency, of seven dependent products (some 5000 cycles each: 16 MMAs 2200,
// GELU 1500, the hand-over) and of the update.  Two epochs of 8192 rows in minibatches of 512
// take 1.37 ms (34 us a minibatch, and the host's first shuffle and copies).
// Before: one launch per product, transposition, reduction and update 8.18 ms; clusters of
// four that exchanged activations through L2 2.65 ms; pieces stored into all eight CTAs by
// st.shared::cluster and a cluster barrier (4400 cycles a hand-over), and weight gradients
// that gathered their operands with 16-byte copies and read the moments in the epilogue
// (35000 cycles) 2.22 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "chain.cuh"
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
constexpr int PIECE = 128 * FB_N * 2; // a CTA's columns of an A operand: 128 rows x K 32, 8-row groups 512 B apart
constexpr int FB_A = FB_CL * PIECE;   // A: 128 rows x K 256
constexpr int FB_B = 4 * FB_N * 64 * 2;
constexpr int FB_SMEM = 2 * FB_A + FB_B;
constexpr int DW_T = 512, DW_N = 32, DW_KC = 8;  // threads, columns per CTA, K-chunks of 64 in shared memory
constexpr int DW_C = DW_N / (DW_T / 128);        // columns per thread
constexpr int DW_B_CHUNK = DW_N * 64 * 2;
constexpr int DW_SMEM = DW_KC * (A_CHUNK + DW_B_CHUNK);
static_assert(FB_C == 8 && DW_C == 8, "a thread's columns are one core-matrix row");

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t in_cta(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
// Bulk copies (16-byte aligned, a multiple of 16 bytes) into shared memory, completion on
// an mbarrier next to the destination: from global memory, and into another CTA of the cluster.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void bulk_s2c(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

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

// D (+)= A B^T over `steps` K-steps of 16: A in blocks of a_k steps and a_bytes bytes with 8-row
// groups a_sbo bytes apart, B in chunks of 4 steps and R_B rows.
template <int R_B>
__device__ __forceinline__ void issue_mma(uint32_t tmem, uint32_t a0, int a_k, uint32_t a_bytes, uint32_t a_sbo, uint32_t b0,
                                          int steps, uint32_t idesc, bool add)
{
    for (int s = 0; s < steps; ++s)
        tc_mma_f16(tmem, smem_desc(a0 + s / a_k * a_bytes + s % a_k * 256, 128, a_sbo),
                   smem_desc(b0 + (s >> 2) * (R_B * 128) + (s & 3) * 256, 128, 1024), idesc, (add || s > 0) ? 1u : 0u);
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// FB_C = 8 values of a row, consecutive columns, as one 16-byte core-matrix row
__device__ __forceinline__ void put8(const float h[FB_C], uint8_t* dst)
{
    *reinterpret_cast<uint4*>(dst) = make_uint4(pack2(h[0], h[1]), pack2(h[2], h[3]), pack2(h[4], h[5]), pack2(h[6], h[7]));
}
// The transposed activations and gradients as the weight-gradient kernel's operands: tiles of
// 128 columns c (rows of dZ^T, H^T) x 64 rows r of the minibatch (K), each in the canonical
// layout (16 KB, contiguous); nk tiles along K.  Element index of (c, r).
__device__ __forceinline__ int64_t t_index(int c, int64_t r, int64_t nk)
{
    return ((int64_t)(c >> 7) * nk + (r >> 6)) * (A_CHUNK / 2) + ((c & 127) >> 3) * 512 + ((r & 63) >> 3) * 64 +
           (c & 7) * 8 + (r & 7);
}
__device__ __forceinline__ void store_t8(const float h[FB_C], __nv_bfloat16* tr, int64_t nk, int64_t r, int c)
{
    __nv_bfloat16* p = tr + t_index(c, r, nk);  // c is a multiple of 8
#pragma unroll
    for (int i = 0; i < FB_C; ++i) p[8 * i] = __float2bfloat16_rn(h[i]);
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
    __shared__ __align__(8) uint64_t mbar, xbar[2];
    __shared__ uint32_t tmem_base;
    __shared__ float red[4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t row0 = (int64_t)blockIdx.x * 128;
    const int y = blockIdx.y, n0 = y * FB_N;
    const uint32_t uA = smem_u32(smem), uB = uA + 2 * FB_A, mb = smem_u32(&mbar), ux = smem_u32(xbar);
    const int lr = 32 * (warp & 3) + lane;  // this thread's row of the tile
    const int c0 = FB_C * (warp >> 2);      // and first column of its slice
    const int64_t r = row0 + lr;
    const bool live = r < g.rows;
    const int64_t nk = (g.rows + 63) / 64;
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_base), FB_N);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(mb, 1);
        mbar_init(ux, 1);
        mbar_init(ux + 8, 1);
    }
    cluster_arrive();  // (waited for before the first copy into another CTA: its barriers are there by then)
    chain_wait();
    chain_next();
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
        *reinterpret_cast<uint4*>(smem + (xr >> 3) * 512 + part * 128 + (xr & 7) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        if (y == 1 && gr < g.rows) {
            __nv_bfloat16* t = g.Xt + t_index(8 * part, gr, nk);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
                t[16 * i] = h.x;
                t[16 * i + 8] = h.y;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base, trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
    uint32_t phase = 0, xph = 0;  // xph bit b: parity of xbar[b]
    bool ok = true;
    // The A operand alternates between two buffers.  A CTA writes its piece of the next one in
    // its own shared memory and copies it into the other CTAs'; `other` bytes arrive from them.
    // No other hand-shake is needed: a piece for a buffer is sent only after a product whose
    // operand held every CTA's previous piece, sent after that CTA's last product from
    // this buffer; and a piece's source is written again only after products of all its readers.
    auto send = [&](uint32_t at, uint32_t bytes, int b, int peers) {  // to the CTAs 0 .. peers - 1
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        const int p = tid - 32;  // (not the thread that issues the MMAs)
        if (p >= 0 && p < peers && p != y) bulk_s2c(in_cta(at, p), at, bytes, in_cta(ux + 8 * b, p));
    };
    // The operands have been issued: wait for them (the `other` bytes of A in buffer b from other CTAs too),
    // multiply, wait for the product.  A wait that gives up leaves the rest of the tile's
    // products out; every barrier is still met, and the pieces that arrive all the same are
    // counted for a last wait: they may not land in the shared memory of a CTA that has left.
    uint32_t late = 0, owed[2] = {0, 0};  // thread 0: bit b: the wait on xbar[b] gave up; bytes not waited for since
    auto multiply = [&](int b, uint32_t other, int steps, uint32_t a_sbo, int N) {
        if (tid == 0 && other) {
            if (ok)
                mbar_expect_tx(ux + 8 * b, other);
            else
                owed[b] += other;
        }
        cp_wait_all();
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (tid == 0 && ok) {
            if (!other || mbar_wait_bounded(ux + 8 * b, (xph >> b) & 1u, MBAR_WAIT_LIMIT)) {
                tc_fence_after();
                issue_mma<FB_N>(tmem, uA + b * FB_A, 2, PIECE, a_sbo, uB, steps, idesc_bf16_f32(128, N), false);
                tc_commit(mb);
            } else {
                late |= 1u << b;
            }
        }
        if (other && ok) xph ^= 1u << b;
        bool w = true;
        if (ok) w = mbar_wait_bounded(mb, phase, MBAR_WAIT_LIMIT);
        phase ^= 1u;
        ok = __syncthreads_and(ok && w);
        tc_fence_after();
    };
    constexpr uint32_t OTHERS = (FB_CL - 1) * PIECE, DY_BYTES = 128 * 16 * 2;
    uint8_t* piece = smem + y * PIECE + (lr >> 3) * 512 + (c0 >> 3) * 128 + (lr & 7) * 16;  // this thread's 16 bytes
    float dg[3][FB_C];  // GELU'(Z) of this thread's values
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        multiply(l & 1, l == 0 ? 0u : OTHERS, l == 0 ? 2 : 16, 512, FB_N);
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
        const int nb = (l + 1) & 1;
        put8(h, piece + nb * FB_A);
        if (l == 0) cluster_wait();
        send(uA + nb * FB_A + y * PIECE, PIECE, nb, l < 2 ? FB_CL : 1);  // (layer 4 is the first CTA's)
        // what only the backward pass and the weight gradients read, while the pieces are on their way
        if (live) store_t8(h, g.Ht[l], nk, r, n0 + c0);
#pragma unroll
        for (int i = 0; i < FB_C; ++i)
            dg[l][i] = 0.5f * e[i] + z[i] * expf(-0.5f * z[i] * z[i]) * 0.39894228040143268f;
    }
    // layer 4 (one CTA of the cluster), the loss and its gradient
    if (y == 0) {
        multiply(1, OTHERS, 16, 512, dout_p(3));
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
            put8(d, smem + (lr >> 3) * 256 + (c0 >> 3) * 128 + (lr & 7) * 16);  // K 16: 8-row groups 256 B apart
            if (live) store_t8(d, g.dYt, nk, r, c0);
            if (c0 == 0) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
                if (lane == 0) red[warp] = loss;
            }
        }
        send(uA, DY_BYTES, 0, FB_CL);
        if (tid == 0) g.loss_part[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
    } else {
        load_operand<FB_N, FB_T>(uB, g.Wt[3], dout_p(3), n0, NH, 0, dout_p(3), 1);
        cp_commit();
    }
    // backward: dZ_l = (dZ_{l+1} W_{l+1}) GELU'(Z_l)
#pragma unroll
    for (int l = 2; l >= 0; --l) {
        multiply(l & 1, l < 2 ? OTHERS : y == 0 ? 0u : DY_BYTES, l == 2 ? 1 : 16, l == 2 ? 256 : 512, FB_N);
        if (l > 0) {
            load_operand<FB_N, FB_T>(uB, g.Wt[l], NH, n0, NH, 0, NH, 4);
            cp_commit();
        }
        float v[FB_C];
        tmem_ld8(trow, v);
#pragma unroll
        for (int i = 0; i < FB_C; ++i) v[i] *= dg[l][i];
        if (l > 0) {
            const int nb = (l - 1) & 1;
            put8(v, piece + nb * FB_A);
            send(uA + nb * FB_A + y * PIECE, PIECE, nb, FB_CL);
        }
        if (live) store_t8(v, g.dZt[l], nk, r, n0 + c0);
    }
    if (!ok && tid == 0) {
        atomicExch(g.err, 1);
        // a last bounded chance for the tensor core before its memory is freed
        mbar_wait_bounded(mb, 0u, MBAR_WAIT_LIMIT);
        mbar_wait_bounded(mb, 1u, MBAR_WAIT_LIMIT);
        // and for the pieces on their way here, if a phase that gave up completes at all
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint32_t next = (xph >> b) & 1u;
            if (((late >> b) & 1u) && !mbar_wait_bounded(ux + 8 * b, next ^ 1u, MBAR_WAIT_LIMIT)) continue;
            if (owed[b] == 0u) continue;
            mbar_expect_tx(ux + 8 * b, owed[b]);
            mbar_wait_bounded(ux + 8 * b, next, MBAR_WAIT_LIMIT);
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive();  // no copy of the cluster is still reading this CTA's shared memory
    cluster_wait();
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
    const __nv_bfloat16* p = l == 3 ? g.dYt : g.dZt[l];
    const int64_t nk = (g.rows + 63) / 64;
    float s = 0.0f;
#pragma unroll 8
    for (int64_t k = lane; k < g.rows; k += 32) s += __bfloat162float(p[t_index(o, k, nk)]);
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
// each of layers 2 and 3, layer 4's 8); the CTAs after them sixteen bias rows each.
__global__ void __launch_bounds__(DW_T, 1) mlp_dw_kernel(TrainArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t mbar, full;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int t = blockIdx.x, l = 0;
    if (t >= DW_TILES) {
        chain_wait();
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
    const uint32_t uA = smem_u32(smem), uB = uA + DW_KC * A_CHUNK, mb = smem_u32(&mbar), uf = smem_u32(&full);
    const int64_t nk = (g.rows + 63) / 64;
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_base), DW_N);
        tmem_relinquish();
    }
    // up to DW_KC K-chunks: A's are contiguous (16 rows of layer 4's), B's are 32 of a tile's 128 rows
    auto fetch = [&](int64_t k0, int nc) {
        const uint32_t ab = l == 3 ? 2048u : (uint32_t)A_CHUNK;
        const __nv_bfloat16* a = A + t_index(m0, k0, nk);
        const __nv_bfloat16* b = B + t_index(n0, k0, nk);
        mbar_expect_tx(uf, nc * (ab + DW_B_CHUNK));
        if (l < 3) bulk_g2s(uA, a, nc * A_CHUNK, uf);
        for (int c = 0; c < nc; ++c) {
            if (l == 3) bulk_g2s(uA + c * A_CHUNK, a + c * (A_CHUNK / 2), ab, uf);
            bulk_g2s(uB + c * DW_B_CHUNK, b + c * (A_CHUNK / 2), DW_B_CHUNK, uf);
        }
    };
    chain_wait();
    chain_next();
    const auto chunks = [&](int64_t k0) { return (int)min((int64_t)DW_KC, nk - k0 / 64); };
    if (tid == 0) {
        mbar_init(mb, 1);
        mbar_init(uf, 1);
        fetch(0, chunks(0));
    }
    // this thread's outputs; parameters and moments are loaded while the operands arrive
    const int o = m0 + 32 * (warp & 3) + lane, c = n0 + DW_C * (warp >> 2);
    const int64_t at = (int64_t)o * din_p(l) + c;
    const bool mine = o < dout_p(l), update = mine && g.adam;
    float p[DW_C], m[DW_C], v[DW_C];
    auto load8 = [&](const float* src, float (&x)[DW_C]) {
#pragma unroll
        for (int i = 0; i < DW_C; i += 4) {
            const float4 q = update ? *reinterpret_cast<const float4*>(src + at + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            x[i] = q.x, x[i + 1] = q.y, x[i + 2] = q.z, x[i + 3] = q.w;
        }
    };
    auto store8 = [&](float* dst, const float (&x)[DW_C]) {
#pragma unroll
        for (int i = 0; i < DW_C; i += 4)
            *reinterpret_cast<float4*>(dst + at + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
    };
    load8(g.W[l], p);
    load8(g.mW[l], m);
    load8(g.vW[l], v);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    uint32_t phase = 0;
    bool ok = true;
    for (int64_t k0 = 0; k0 < g.rows && ok; k0 += 64 * DW_KC) {
        if (tid == 0) {
            if (k0 > 0) fetch(k0, chunks(k0));
            if (mbar_wait_bounded(uf, phase, MBAR_WAIT_LIMIT)) {
                tc_fence_after();
                issue_mma<DW_N>(tmem, uA, 4, A_CHUNK, 1024, uB, (int)min((int64_t)64 * DW_KC, g.rows - k0) / 16,
                                idesc_bf16_f32(128, DW_N), k0 > 0);
                tc_commit(mb);
            }
        }
        ok = mbar_wait_bounded(mb, phase, MBAR_WAIT_LIMIT);
        phase ^= 1u;
        ok = __syncthreads_and(ok);
    }
    tc_fence_after();
    if (ok) {
        float d[DW_C];
        tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(DW_C * (warp >> 2)), d);
        if (mine && !g.adam) store8(g.gW[l], d);
        if (update) {
#pragma unroll
            for (int i = 0; i < DW_C; ++i) p[i] = adam_step(p[i], d[i], m[i], v[i], g);
            store8(g.W[l], p);
            store8(g.mW[l], m);
            store8(g.vW[l], v);
            put8(p, reinterpret_cast<uint8_t*>(g.Wb[l] + at));
#pragma unroll
            for (int i = 0; i < DW_C; ++i) g.Wt[l][(int64_t)(c + i) * dout_p(l) + o] = __float2bfloat16_rn(p[i]);
        }
    } else if (tid == 0) {
        atomicExch(g.err, 1);
        // a last bounded chance for the copies in flight and the tensor core
        mbar_wait_bounded(uf, phase ^ 1u, MBAR_WAIT_LIMIT);
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
    e = launch_chained(mlp_fb_kernel, dim3((unsigned)((g.rows + 127) / 128), FB_CL), FB_T, FB_SMEM, s, g);
    if (e != cudaSuccess) return e;
    return launch_chained(mlp_dw_kernel, DW_TILES + BIAS_ROWS / (DW_T / 32), DW_T, DW_SMEM, s, g);
}

}  // namespace ptadd
