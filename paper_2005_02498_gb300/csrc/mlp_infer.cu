// mlp_infer.cu -- fused surrogate inference: raw closure inputs -> sym(Lp),
// the whole 30 -> 256 -> 256 -> 256 -> 6 network in one persistent kernel.
//
// A pair of CTAs (a cluster of 2, one CTA per SM) walks pairs of 128-row tiles of the input.
// The tensor cores of the two SMs work as one (cta_group::2: M = 256, the rows of both
// tiles; each SM holds its own rows of A and D and half of the rows of every weight), so
// that all weights stay in shared memory: 64 KB per hidden layer and CTA.  Each CTA has
// 18 warps in three roles:
//   * warps 0-15 ("epilogue warps"): per tile they map and standardise the
//     raw features (sigma / 200 MPa, log10(rho + 1e10)) into the FP16
//     layer-1 operand (and its rounding residual, for the trust region), test
//     the box of the trust region, and run the epilogues: accumulator -> GELU ->
//     FP16 activations in shared memory, 64 columns at a time (warp w: TMEM
//     lanes 32 (w mod 4) .. +31, i.e. its rows, and 16 columns), the Mahalanobis
//     test, and the de-standardised FP64 outputs.  The map of tile t + 1 runs after
//     tile t's second hidden epilogue, beside layer 3; its features were loaded into
//     registers, coalesced, a tile ahead;
//   * warp 16, lane 0 of the first CTA ("MMA issuer"): issues every tcgen05 MMA of the
//     pair, each K-slice as soon as its activation chunk is in both shared
//     memories, and never waits for an MMA to finish;
//   * warp 17, lane 0: copies the CTA's resident operands in, once (three bulk copies
//     from a copy laid out in global memory when the parameters or maps change).
// What bounds it: the chain through one tile.  A layer's MMAs take 2450 cycles (17 of
// 256 x 256 x 16), its GELUs 2000 (the special-function unit: 128 x 256 tanh at 16 per
// clock), and only the part after the first chunk of a layer overlaps; the activations of a
// second pair of tiles would not fit beside the weights.  10^6 rows take 392 us.  One CTA
// per tile with weights streamed from L2 through two 32 KB stages took 468 us: a stage came
// back to the issuer some 1700 cycles after its commit, so a layer took 4300 cycles
// at any copy rate.  Seven 16 KB stages (528 us) and two tiles in flight per SM (477 us) did not help.
// Trust region: the distance d2 = |L^-1 z|^2 is a 128 x 32 x 32 product,
// W = Z L^-T, that the tensor core computes next to layer 1 (into 32 spare
// columns of the second accumulator) in split FP16: z = z_hi + z_lo with
// z_hi the layer-1 operand itself, s L^-1 = L_hi + L_lo with s a power of
// two that brings max |L^-1| to [2^13, 2^14), and W = z_hi L_hi + z_hi L_lo +
// z_lo L_hi (the dropped z_lo L_lo term is ~2^-22 relative).  The epilogue
// warps of the first column slice read their row of W once layer 1 is done
// and sum w_i^2 / s^2 in FP32.
// Two TMEM accumulators of 256 columns alternate between the layers (1 -> A,
// 2 -> B, 3 -> A, 4 -> B), and the activations of a layer are handed over in
// 64-column chunks, each with its own mbarrier: while the epilogue warps turn
// chunk c + 1 of layer l's accumulator into activations, the tensor core
// already runs layer l + 1 on chunk c (its K-slice 64 c .. 64 c + 63).  So
// the GELU work of a layer runs beside the next layer's MMAs instead of
// between them.  Barriers of the pair, in the first CTA, one arrival per epilogue warp of
// both: xbar (layer-1 operand ready), hbar[4] (activation chunk ready; it cannot run two
// phases ahead of the MMA issuer, because its next phase needs the next layer's
// accumulator, which needs this phase), wbar (W2 and W3 are there).  In each CTA:
// accbar[4] (layer l's MMAs complete, tcgen05.commit to both CTAs; one barrier per layer,
// because layer 1 of the next tile may complete before the epilogue has waited for layer 4
// of this one), lxbar (this CTA's box tests).  The arrivals at the other CTA carry the
// default (CTA) scope: what they hand over is this CTA's own shared memory, which the
// writing lanes have already made visible to the tensor core's proxy; a release at
// cluster scope waits for the thread's outputs on their way to global memory (557 us).
// Every wait has an iteration limit; a wait that gives up raises the abort flags of both
// CTAs, every role leaves its loop, the MMA issuer waits (bounded) for its last MMAs and
// warp 17 for its copies, and after a barrier of the cluster the kernel frees its tensor
// memory and sets the error flag.
//
// Operands are FP16 (the trained weights are BF16, which FP16 holds exactly
// in its normal range; activations and inputs are rounded to FP16, relative
// step 2^-11), accumulators FP32.  GELU here is 0.5 z (1 + erf(z / sqrt 2))
// with erf(x) ~ tanh(x (A + B x^2)), A = 1.12967582605, B = 0.0997927024 (a
// minimax fit of erf on [0, 6] made for this kernel; |error| <= 2.8e-4), the
// tanh by the hardware f16x2 approximation, and the whole activation in f16x2
// arithmetic: the kernel stores a' = z (1 + tanh(u)) = 2 GELU(z) and takes
// the factor 1/2 into the next layer's weights (W2, W3, W4 are scaled by 1/2
// when they are staged, exactly).  Every hidden layer's bias is already in
// its accumulator, split into two FP16 parts (b_hi = fp16(b), b_lo = fp16(b -
// b_hi)): layer 1's rides in the two padding columns of its K = 32 operand
// (inputs 1 there, W1's columns the bias), layers 2 and 3 start with one
// K = 16 MMA of a constant operand (1 in K columns 0 and 1) against a bias
// block whose K columns 0, 1 (layer 2) or 2, 3 (layer 3) hold the two parts; the eight equal
// rows of the constant operand are read at a stride of zero.  So an activation pair costs
// one conversion, four f16x2 FMA-pipe operations and one special-function
// operation.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "ptadd_internal.cuh"
#include "tc_gemm.cuh"

namespace ptadd {

namespace {

constexpr int EW = 16;             // epilogue warps
constexpr int IT = 32 * EW;        // epilogue threads (rows per tile: 128)
constexpr int IT_ALL = IT + 64;    // + the MMA warp and the warp that copies the resident operands in
constexpr int NF = 30, NO = 6;
constexpr int X_BYTES = 128 * 32 * 2;   // layer-1 A operand (FP16) or its residual, SBO 512
constexpr int H_BYTES = 128 * 256 * 2;  // hidden activations, SBO 4096
// the B operands: this CTA's half of the rows (output columns) of each
constexpr int W1_BYTES = 128 * 32 * 2;   // SBO 512
constexpr int WH_BYTES = 128 * 256 * 2;  // W2 / 2 or W3 / 2, SBO 4096
constexpr int W4_BYTES = 8 * 256 * 2;    // SBO 4096
constexpr int LI_BYTES = 16 * 32 * 2;    // L_hi or L_lo: rows (i) x 32 K (j), SBO 512
constexpr int BB_BYTES = 128 * 8 * 2;    // biases of layers 2 and 3: K columns 0, 1 and 2, 3 (two FP16 parts each), SBO 128
constexpr int ONES_BYTES = 8 * 16 * 2;   // A operand of a bias MMA: 8 equal rows, 1 in the layer's two K columns, else 0
constexpr int MAHA_COL = 288;            // TMEM columns of W (second accumulator, clear of layer 4's 16)
// maps as the kernel keeps them (floats): xm, 1/xs, ym, ys, box lo, box hi, d2 threshold, 1/s^2, layer 4's bias
constexpr int NV_XM = 0, NV_XR = NV_XM + NF, NV_YM = NV_XR + NF, NV_YS = NV_YM + NO, NV_LO = NV_YS + NO,
              NV_HI = NV_LO + NF, NV_THR = NV_HI + NF, NV_S2 = NV_THR + 1, NV_B4 = NV_S2 + 1, NV_COUNT = NV_B4 + 16;
constexpr int NV_BYTES = (NV_COUNT * 4 + 127) / 128 * 128;
// what stays in shared memory, laid out in global memory as it is there, one block per
// CTA of a pair: three bulk copies (what layer 1 needs, then W2, then W3)
constexpr int R_W1 = 0;
constexpr int R_LH = R_W1 + W1_BYTES;
constexpr int R_LL = R_LH + LI_BYTES;
constexpr int R_W4 = R_LL + LI_BYTES;
constexpr int R_BB = R_W4 + W4_BYTES;
constexpr int R_ONES = R_BB + BB_BYTES;  // layer 2's, then layer 3's
constexpr int R_NV = R_ONES + 2 * ONES_BYTES;
constexpr int R_WH = R_NV + NV_BYTES;    // W2, then W3
constexpr int RES_BYTES = R_WH + 2 * WH_BYTES;
constexpr int OFF_X = 0;                  // z_hi
constexpr int OFF_XLO = OFF_X + X_BYTES;  // z_lo, the same layout
constexpr int OFF_H = OFF_XLO + X_BYTES;
constexpr int OFF_RES = OFF_H + H_BYTES;
constexpr int OFF_BOX = OFF_RES + RES_BYTES;  // box test per row [2 tiles][128]
constexpr int INFER_SMEM = OFF_BOX + 2 * 128;
static_assert(R_WH % 128 == 0 && RES_BYTES % 16 == 0, "bulk copies need 16-byte alignment");
static_assert(INFER_SMEM + 512 <= 232448, "shared memory of one CTA, the barriers included");
// raw features of a tile: 128 rows x 15 pairs, pair e = tid + IT i in thread tid's slot i
constexpr int FPT = (128 * NF / 2 + IT - 1) / IT;

__device__ __forceinline__ uint32_t canon(int r, int k, int sbo)
{
    return (uint32_t)((r >> 3) * sbo + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// ------------------------------------------------ PTX of a CTA pair
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// all threads of both CTAs
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// a shared-memory address of this CTA, in the CTA of rank r of the cluster
__device__ __forceinline__ uint32_t in_cta(uint32_t addr, uint32_t r)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(r));
    return a;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
// One MMA of the pair, M = 256: the operands lie at the same shared-memory addresses in
// both CTAs, A's rows 0..127 and B's first N / 2 rows in the first CTA, the others in the
// second; each CTA's tensor memory gets its 128 rows of D, all N columns.
__device__ __forceinline__ void tc_mma2_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// completion of the MMAs issued so far, on the barrier at this address in both CTAs
__device__ __forceinline__ void tc_commit2(uint32_t mbar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(mbar),
        "h"((uint16_t)3)
        : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
// bytes (a multiple of 16, both addresses 16-byte aligned) from global to shared, completion on mbar
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(mbar)
                 : "memory");
}
// Two consecutive raw features, loaded ahead of use: asm volatile, so that the
// compiler leaves the load where it is.  One 16-byte load where the array is 16-byte
// aligned (every pair then is).
__device__ __forceinline__ void load_pair(const double* p, bool wide, double f[2])
{
    asm volatile(
        "{\n .reg .pred w;\n setp.ne.b32 w, %3, 0;\n @w ld.global.nc.v2.f64 {%0, %1}, [%2];\n"
        " @!w ld.global.nc.f64 %0, [%2];\n @!w ld.global.nc.f64 %1, [%2 + 8];\n}\n"
        : "=&d"(f[0]), "=&d"(f[1])
        : "l"(p), "r"((int)wide));
}

// 2 GELU(z) of two values in f16x2 (see the header for the approximation)
__device__ __forceinline__ uint32_t gelu2x2_f16(float2 z)
{
    const __half2 h = __floats2half2_rn(z.x, z.y);
    const __half2 z2 = __hmul2(h, h);
    const __half2 u = __hmul2(h, __hfma2(z2, __float2half2_rn(0.03528185f), __float2half2_rn(0.79880562f)));
    uint32_t t;  // K3 = B / (2 sqrt 2), K1 = A / sqrt 2
    asm("tanh.approx.f16x2 %0, %1;" : "=r"(t) : "r"(*reinterpret_cast<const uint32_t*>(&u)));
    const __half2 g = __hfma2(h, *reinterpret_cast<const __half2*>(&t), h);
    return *reinterpret_cast<const uint32_t*>(&g);
}

// 16 consecutive FP32 columns of this thread's TMEM lane, without waiting:
// the registers hold the values only after tmem_wait_ld16 on them.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// Waits for every load issued so far; the loaded registers pass through the
// statement, so that no use of them is scheduled before it.
__device__ __forceinline__ void tmem_wait_ld16(uint32_t r[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// Accumulator values (16 columns; the bias is in them) -> 2 GELU as 8 f16x2 words.
__device__ __forceinline__ void gelu16(const uint32_t r[16], uint32_t w[8])
{
#pragma unroll
    for (int i = 0; i < 8; ++i)
        w[i] = gelu2x2_f16(make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])));
}
// ... into H (row, columns c0 .. c0 + 15)
__device__ __forceinline__ void store16(const uint32_t w[8], int row, int c0, uint8_t* sH)
{
    *reinterpret_cast<uint4*>(sH + canon(row, c0, 4096)) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(sH + canon(row, c0 + 8, 4096)) = make_uint4(w[4], w[5], w[6], w[7]);
}
// Two consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float v[2])
{
    uint32_t r0, r1;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    v[0] = __uint_as_float(r0);
    v[1] = __uint_as_float(r1);
}

// 8 BF16 values -> 8 FP16 values times a power of two (exact in FP16's normal range)
__device__ __forceinline__ uint4 bf16x8_to_f16x8(uint4 v, float scale)
{
    uint32_t in[4] = {v.x, v.y, v.z, v.w}, out[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&in[i]));
        const __half2 h = __floats2half2_rn(f.x * scale, f.y * scale);
        out[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(out[0], out[1], out[2], out[3]);
}

// FP64 -> FP32 (round to nearest even; results below FP32's normal range become
// zeros, which no caller can tell from them) and FP32 -> FP64 (exact) on the integer
// pipe: the conversion instructions run on the FP64 pipe, 2 lanes per clock on this GPU,
// and are issued even where a select discards their result.
__device__ __forceinline__ float d2f_rn(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7FFu, sign = hi & 0x80000000u;
    uint32_t f = ((e - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
    const uint32_t rest = lo & 0x1FFFFFFFu;  // the 29 dropped bits
    f += (rest > 0x10000000u || (rest == 0x10000000u && (f & 1u))) ? 1u : 0u;  // carries into the exponent
    if (e < 897u) f = 0u;
    if (e > 1150u) f = (e == 0x7FFu && ((hi & 0xFFFFFu) | lo)) ? 0x7FFFFFFFu : 0x7F800000u;
    return __uint_as_float(sign | f);
}
__device__ __forceinline__ double f2d(float x)
{
    const uint32_t u = __float_as_uint(x), sign = u & 0x80000000u;
    uint32_t m = u & 0x7FFFFFu, e = (u >> 23) & 0xFFu;
    if (e == 0u && m) {  // subnormal
        const int up = __clz((int)m) - 8;
        m = (m << up) & 0x7FFFFFu;
        e = (uint32_t)(897 - up);
    } else {
        e = e == 0u ? 0u : e == 0xFFu ? 0x7FFu : e + 896u;
    }
    return __hiloint2double((int)(sign | (e << 20) | (m >> 3)), (int)(m << 29));
}

// Bounded wait on an mbarrier phase that also gives up when another role of the pair
// has raised the abort flag: false if the phase did not complete.
__device__ __forceinline__ bool wait_or_abort(uint32_t mbar, uint32_t parity, volatile int* abort_flag)
{
    const long long t0 = clock64();
    while (!mbar_try_wait(mbar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > MBAR_WAIT_LIMIT) return false;
    }
    return true;
}

// Features k (even) and k + 1 from the FP64 input rounded to FP32: sigma / 200 MPa (k < 6)
// or log10(rho + 1e10), less the mean, times the reciprocal deviation; all FP32 arithmetic
// (the FP64 pipe is slow on this part).  Every rounding is written out, because a
// last-bit difference here can flip the operand's FP16 rounding: the product by log10(2) is
// rounded before the subtraction, except in columns 6 and 7 of each 8, where the two
// are one fused operation.  That split has no reason in the mathematics; it is kept because the
// trust-region flags depend on it: with every column fused 2 to 9 of 10^6 flags change (8 sets
// of inputs), and the rates by 6e-5.
__device__ __forceinline__ float standardise(double v, int k, float mean, float rdev)
{
    constexpr float LOG10_2 = 0.30102999566398120f;
    const float x = d2f_rn(v);
    float c;
    if (k < 6) {
        c = __fsub_rn(__fmul_rn(x, (float)(1.0 / 200e6)), mean);
    } else {
        const float l = __log2f(x + 1e10f);
        c = (k & 7) == 6 ? fmaf(l, LOG10_2, -mean) : __fsub_rn(__fmul_rn(l, LOG10_2), mean);
    }
    return __fmul_rn(c, rdev);
}

struct InferArgs {
    const double* feat;  // [n x 30]
    int64_t n;
    int feat_wide;       // feat is 16-byte aligned
    const uint8_t* res;  // [2][RES_BYTES]: what stays in shared memory, per CTA of a pair
    double* lp6;         // [n x 6]
    uint8_t* in_region;  // [n] or null
    int* err;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(IT_ALL, 1) mlp_infer_kernel(InferArgs g)
{
    // every region below starts at a multiple of 16 bytes, all the no-swizzle
    // operand layouts need; pointers derived from the array itself keep the
    // compiler's shared-memory address space (plain shared loads and stores)
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t xbar, lxbar, hbar[4], accbar[4], wbar, drainbar, resbar, whbar;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    uint8_t* base = smem_raw;
    uint8_t* sX = base + OFF_X;
    uint8_t* sXlo = base + OFF_XLO;
    uint8_t* sH = base + OFF_H;
    uint8_t* sBox = base + OFF_BOX;
    const float* snv = reinterpret_cast<const float*>(base + OFF_RES + R_NV);
    const uint32_t uX = smem_u32(sX), uXlo = smem_u32(sXlo), uH = smem_u32(sH);
    const uint32_t uR = smem_u32(base + OFF_RES);
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t rank = cluster_rank();
    const int64_t n_pairs = (g.n + 255) / 256, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    // (no CTA leaves early: the grid has no more pairs than the input)
    const int64_t my_tiles = (n_pairs - 1 - pair) / pairs + 1;
    // each mbarrier is 8 bytes: barrier k of an array at u0 + 8 k
    const uint32_t ux = smem_u32(&xbar), ulx = smem_u32(&lxbar), uacc0 = smem_u32(accbar), uh0 = smem_u32(hbar);
    const uint32_t ures = smem_u32(&resbar), uwh = smem_u32(&whbar), uw = smem_u32(&wbar), udrain = smem_u32(&drainbar);
    const uint32_t uabort = smem_u32(const_cast<int*>(&abort_flag));

    if (warp == 0) tmem_alloc2(smem_u32(&tmem_base), 512);
    if (tid == 0) {
        abort_flag = 0;
        mbar_init(ux, 2 * EW);
        mbar_init(ulx, EW);
        for (int c = 0; c < 4; ++c) mbar_init(uh0 + 8 * c, 2 * EW);
        for (int l = 0; l < 4; ++l) mbar_init(uacc0 + 8 * l, 1);
        mbar_init(uw, 2);
        mbar_init(udrain, 1);
        mbar_init(ures, 1);
        mbar_init(uwh, 1);
    }
    if (tid < 256) sBox[tid] = 1;
    // the bias columns of the layer-1 operand (inputs 1 there, residual 0) stay as they are
    if (tid < 128) {
        *reinterpret_cast<uint32_t*>(sX + canon(tid, NF, 512)) = 0x3c003c00u;
        *reinterpret_cast<uint32_t*>(sXlo + canon(tid, NF, 512)) = 0u;
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the barrier inits and both halves of the tensor memory are there
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    bool ok = true;
    auto raise_abort = [&]() {  // in both CTAs
        for (uint32_t r = 0; r < 2; ++r)
            asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(in_cta(uabort, r)), "r"(1) : "memory");
    };

    if (warp == EW + 1) {
        // ------------------------------------------------ the resident operands
        if ((tid & 31) == 0) {
            const uint8_t* res = g.res + (size_t)rank * RES_BYTES;
            mbar_expect_tx(ures, R_WH);
            bulk_g2s(uR, res, R_WH, ures);
            mbar_expect_tx(uwh, 2 * WH_BYTES);
            bulk_g2s(uR + R_WH, res + R_WH, WH_BYTES, uwh);
            bulk_g2s(uR + R_WH + WH_BYTES, res + R_WH + WH_BYTES, WH_BYTES, uwh);
            // (no copy may still be landing when the CTA leaves: both are waited for, bounded)
            if (!mbar_wait_bounded(ures, 0u, MBAR_WAIT_LIMIT) || !mbar_wait_bounded(uwh, 0u, MBAR_WAIT_LIMIT)) {
                raise_abort();
                atomicExch(g.err, 1);
            }
            mbar_arrive_cluster(in_cta(uw, 0));
        }
    } else if (warp == EW) {
        // ------------------------------------------------ MMA issuer of the pair
        if (rank == 0 && (tid & 31) == 0) {
            const uint32_t id_h = idesc_f16_f32(256, 256), id_o = idesc_f16_f32(256, 16);
            const uint32_t id_m = idesc_f16_f32(256, 32);
            const uint32_t accA = tmem, accB = tmem + 256;
            uint32_t xph = 0, hph = 0;  // hph bit kc: parity of hbar[kc]
            bool mma_out = false;       // MMAs issued (for the abort path)
            auto chunk = [&](int kc) {  // activation chunk kc of the current layer is ready
                const bool w = wait_or_abort(uh0 + 8 * kc, (hph >> kc) & 1u, &abort_flag);
                hph ^= 1u << kc;
                tc_fence_after();
                return w;
            };
            // trust region: W = z_hi L_hi + z_hi L_lo + z_lo L_hi (kind::f16 with FP16 operands),
            // as soon as the tile's input map is ready
            auto trust = [&]() {
                const bool w = wait_or_abort(ux, xph, &abort_flag);
                xph ^= 1u;
                if (!w) return false;
                tc_fence_after();
                for (int s = 0; s < 2; ++s) {
                    const uint64_t zh = smem_desc(uX + s * 256, 128, 512), zl = smem_desc(uXlo + s * 256, 128, 512);
                    const uint64_t lh = smem_desc(uR + R_LH + s * 256, 128, 512);
                    const uint64_t ll = smem_desc(uR + R_LL + s * 256, 128, 512);
                    tc_mma2_f16(tmem + MAHA_COL, zh, lh, id_m, s ? 1u : 0u);
                    tc_mma2_f16(tmem + MAHA_COL, zh, ll, id_m, 1u);
                    tc_mma2_f16(tmem + MAHA_COL, zl, lh, id_m, 1u);
                }
                mma_out = true;
                return true;
            };
            // layer 1: X [128 x 32] W1^T -> A
            auto layer1 = [&]() {
                for (int s = 0; s < 2; ++s)
                    tc_mma2_f16(accA, smem_desc(uX + s * 256, 128, 512), smem_desc(uR + R_W1 + s * 256, 128, 512), id_h,
                                s ? 1u : 0u);
                tc_commit2(uacc0);
            };
            if ((ok = trust())) {
                layer1();
                ok = wait_or_abort(uw, 0u, &abort_flag);
                tc_fence_after();
            }
            for (int64_t it = 0; it < my_tiles && ok; ++it) {
                // layers 2, 3: H [128 x 256] W^T, K-slice by K-slice as soon as the
                // epilogues of both CTAs have written their activation chunk
                for (int l = 1; l <= 2 && ok; ++l) {
                    const uint32_t acc = (l == 1) ? accB : accA, uW = uR + R_WH + (l - 1) * WH_BYTES;
                    for (int kc = 0; kc < 4; ++kc) {
                        if (!(ok = chunk(kc))) break;
                        // the bias first: ones [128 x 16] (b_hi, b_lo, 0..)^T sets the accumulator
                        // (only now: the previous layer's epilogue has read it)
                        if (kc == 0)
                            tc_mma2_f16(acc, smem_desc(uR + R_ONES + (l - 1) * ONES_BYTES, 128, 0),
                                        smem_desc(uR + R_BB, 0, 128), id_h, 0u);
                        for (int k = 4 * kc; k < 4 * kc + 4; ++k)
                            tc_mma2_f16(acc, smem_desc(uH + k * 256, 128, 4096), smem_desc(uW + k * 256, 128, 4096),
                                        id_h, 1u);
                    }
                    if (ok) tc_commit2(uacc0 + 8 * l);
                }
                const bool more = it + 1 < my_tiles;
                // (the second accumulator is free but for layer 4's columns)
                if (ok && more) ok = trust();
                // layer 4: H [128 x 256] W4^T -> B (16 columns, 6 used)
                for (int kc = 0; kc < 4 && ok; ++kc) {
                    if (!(ok = chunk(kc))) break;
                    for (int s = 4 * kc; s < 4 * kc + 4; ++s)
                        tc_mma2_f16(accB, smem_desc(uH + s * 256, 128, 4096), smem_desc(uR + R_W4 + s * 256, 128, 4096),
                                    id_o, s ? 1u : 0u);
                }
                if (!ok) break;
                tc_commit2(uacc0 + 24);
                if (more) layer1();  // (every layer-3 chunk, accumulator A, has been read)
            }
            if (!ok) {
                raise_abort();
                // the tensor cores may still be busy: wait (bounded) for a commit
                // of everything issued before the tensor memory is freed
                if (mma_out) {
                    tc_commit2(udrain);
                    mbar_wait_bounded(udrain, 0u, MBAR_WAIT_LIMIT);
                }
                atomicExch(g.err, 1);
            }
        }
    } else {
        // ------------------------------------------------ epilogue warps
        const int lg = warp & 3, cs = warp >> 2;  // TMEM lane group (rows) and 16-column slice of a chunk
        const int lane = tid & 31, erow = 32 * lg + lane;
        const uint32_t tmem_row = tmem + ((uint32_t)(32 * lg) << 16);
        const uint32_t ux_lead = in_cta(ux, 0), uh_lead = in_cta(uh0, 0);
        uint32_t accph = 0, xph = 0;  // bit l: parity of accbar[l]; of lxbar
        auto wait_acc = [&](int l) {
            const bool w = wait_or_abort(uacc0 + 8 * l, (accph >> l) & 1u, &abort_flag);
            accph ^= 1u << l;
            if (!w) raise_abort();
            tc_fence_after();
            return w;
        };
        // hand this warp's finished share of an operand chunk to the MMA issuer
        auto publish = [&](uint32_t mbar_lead) {
            fence_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mbar_lead);
        };
        auto first_row = [&](int64_t it) { return ((pair + it * pairs) * 2 + rank) * 128; };
        // (the second tile of the last pair may have no rows)
        auto rows_of = [&](int64_t it) { return (int)max((int64_t)0, min((int64_t)128, g.n - first_row(it))); };
        double f[FPT][2];  // raw features of the next tile
        const bool wide = g.feat_wide != 0;
        auto fetch = [&](int64_t it) {
            // unconditional loads (of the first pair where there is nothing to load): a load in
            // a branch is waited for where the branch ends, here a tile too early
            const int np = it < my_tiles ? (NF / 2) * rows_of(it) : 0;
            const double* p = g.feat + first_row(it) * NF;
#pragma unroll
            for (int i = 0; i < FPT; ++i)
                load_pair(tid + IT * i < np ? p + 2 * (tid + IT * i) : g.feat, wide, f[i]);
        };
        // the input map of tile it (its features are in f): the FP16 layer-1 operand z_hi,
        // its residual z_lo and the box test; then the loads for the tile after it
        auto map_tile = [&](int64_t it) {
            const int np = (NF / 2) * rows_of(it);
#pragma unroll
            for (int i = 0; i < FPT; ++i) {
                const int e = tid + IT * i;
                if (e >= 128 * (NF / 2)) break;
                const int row = e / (NF / 2), k = 2 * (e - row * (NF / 2));
                float z[2] = {0.0f, 0.0f};  // rows beyond the input
                if (e < np) {
                    bool box = true;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        z[c] = standardise(f[i][c], k, snv[NV_XM + k + c], snv[NV_XR + k + c]);
                        box = box && z[c] >= snv[NV_LO + k + c] && z[c] <= snv[NV_HI + k + c];
                    }
                    if (!box) sBox[(it & 1) * 128 + row] = 0;
                }
                const __half2 h = __floats2half2_rn(z[0], z[1]);
                const float2 hf = __half22float2(h);
                const __half2 r = __floats2half2_rn(z[0] - hf.x, z[1] - hf.y);
                *reinterpret_cast<__half2*>(sX + canon(row, k, 512)) = h;
                *reinterpret_cast<__half2*>(sXlo + canon(row, k, 512)) = r;
            }
            publish(ux_lead);
            if (lane == 0) mbar_arrive(ulx);  // (this CTA's box tests)
            fetch(it + 1);
        };
        auto outputs = [&](int64_t it) {  // layer 4 -> FP64 outputs (two columns per thread of the last three column slices)
            const int64_t r0 = first_row(it);
            const int valid = rows_of(it);
            if (cs > 0) {
                float v[2];
                tmem_ld2(tmem_row + 256u + (uint32_t)(2 * (cs - 1)), v);
                if (erow < valid) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int o = 2 * (cs - 1) + c;
                        g.lp6[(r0 + erow) * NO + o] = f2d((v[c] + snv[NV_B4 + o]) * snv[NV_YS + o] + snv[NV_YM + o]);
                    }
                }
            }
        };
        fetch(0);
        if (!(ok = wait_or_abort(ures, 0u, &abort_flag))) raise_abort();
        if (ok) map_tile(0);
        for (int64_t it = 0; it < my_tiles && ok; ++it) {
            // 1. hidden layers: activations chunk by chunk, each handed over at once
            for (int l = 0; l < 3 && ok; ++l) {
                ok = wait_acc(l);
                if (!ok) break;
                const uint32_t acc_col = (l == 1) ? 256u : 0u;
                // the load of chunk kc + 1 runs while chunk kc is turned into activations
                uint32_t ra[16], rb[16];
                tmem_ld16_async(tmem_row + acc_col + (uint32_t)(16 * cs), ra);
                if (l == 0 && cs == 0) {
                    // trust region of this row: its row of W lies in columns the
                    // layer-2 MMAs overwrite, so it is read before the first hand-over.
                    // (lxbar, to have seen every warp's box tests; its next phase needs this warp)
                    uint32_t wv[32];
                    tmem_ld16_async(tmem_row + (uint32_t)MAHA_COL, wv);
                    tmem_ld16_async(tmem_row + (uint32_t)MAHA_COL + 16u, wv + 16);
                    if (!(ok = wait_or_abort(ulx, xph, &abort_flag))) raise_abort();
                    xph ^= 1u;
                    tmem_wait_ld16(wv);
                    tmem_wait_ld16(wv + 16);
                    float d2 = 0.0f;
#pragma unroll
                    for (int i = 0; i < NF; ++i) {
                        const float w = __uint_as_float(wv[i]);
                        d2 = fmaf(w, w, d2);
                    }
                    uint8_t* bx = sBox + (it & 1) * 128 + erow;  // this tile's half: the next tile's map
                    const bool box = *bx != 0;                   // may already be writing the other
                    *bx = 1;                                     // (read here only; written again two tiles on)
                    if (erow < rows_of(it) && g.in_region)
                        g.in_region[first_row(it) + erow] = (box && d2 * snv[NV_S2] <= snv[NV_THR]) ? 1 : 0;
                }
                // chunk 0 is handed over at once (the tensor cores wait for it), chunks 1 and 2
                // one step late, after the next chunk's arithmetic, so that the proxy
                // fence finds the stores done (10^6 rows, same build: all late 418 us, all at once 462, so 410)
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    const int c0 = 64 * kc + 16 * cs;
                    uint32_t* cur = (kc & 1) ? rb : ra;
                    uint32_t* nxt = (kc & 1) ? ra : rb;
                    tmem_wait_ld16(cur);
                    if (kc < 3) tmem_ld16_async(tmem_row + acc_col + (uint32_t)(c0 + 64), nxt);
                    uint32_t w[8];
                    gelu16(cur, w);
                    if (kc > 1) publish(uh_lead + 8 * (kc - 1));
                    store16(w, erow, c0, sH);
                    if (kc == 0) publish(uh_lead);
                }
                publish(uh_lead + 24);
                // the next tile's input map, while layer 3 runs (after layer 1's epilogue: 1 % slower)
                if (l == 1 && it + 1 < my_tiles) map_tile(it + 1);
            }
            if (!ok) break;
            // 2. the outputs; the tensor cores are at the next tile's layer 1
            if (!(ok = wait_acc(3))) break;
            outputs(it);
            tc_fence_before();
        }
        if (!ok && lane == 0) atomicExch(g.err, 1);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // no arrival, MMA or flag of the pair is still on its way to this CTA
    if (warp == 0) tmem_dealloc2(tmem, 512);
}

// What the inference kernel keeps in shared memory (RES_BYTES for each CTA of a pair,
// that CTA's half of the rows of every weight): W1 with the bias of layer 1 in K
// columns 30 and 31 (two FP16 parts), s L^-1 in two FP16 parts, W4 / 2, the biases of
// layers 2 and 3 and the ones operands of the bias MMAs, the maps, W2 / 2 and W3 / 2, all
// matrices in the canonical no-swizzle K-major layout (K-adjacent core matrices 128 B
// apart).  Blocks 0 .. 63 lay out W2 and W3, blocks 64 and 65 the rest.
constexpr int WH_BLOCKS = 2 * 256 * 32 / 256;
__global__ void __launch_bounds__(256) tile_resident_kernel(const __nv_bfloat16* __restrict__ W1,
                                                            const float* __restrict__ b1,
                                                            const __nv_bfloat16* __restrict__ W2,
                                                            const float* __restrict__ b2,
                                                            const __nv_bfloat16* __restrict__ W3,
                                                            const float* __restrict__ b3,
                                                            const __nv_bfloat16* __restrict__ W4,
                                                            const float* __restrict__ b4, const float* __restrict__ nv,
                                                            uint8_t* __restrict__ out)
{
    __shared__ unsigned li_max;  // bits of max |L^-1| (non-negative floats order as integers)
    const int tid = threadIdx.x;
    if (blockIdx.x < WH_BLOCKS) {  // one 16-byte group of W2 or W3: row r, group kk
        const int v = blockIdx.x * 256 + tid, l = v >> 13, r = (v >> 5) & 255, kk = v & 31;
        uint8_t* dst = out + (size_t)(r >> 7) * RES_BYTES + R_WH + l * WH_BYTES + canon(r & 127, 8 * kk, 4096);
        *reinterpret_cast<uint4*>(dst) =
            bf16x8_to_f16x8(*reinterpret_cast<const uint4*>((l ? W3 : W2) + r * 256 + 8 * kk), 0.5f);
        return;
    }
    const int rank = blockIdx.x - WH_BLOCKS;
    uint8_t* res = out + (size_t)rank * RES_BYTES;
    if (tid == 0) li_max = 0u;
    __syncthreads();
    const float* gLi = nv + 4 * NF + 2 * NO;  // L^-1, NF x NF row-major, lower triangle
    for (int e = tid; e < NF * NF; e += 256) atomicMax(&li_max, __float_as_uint(fabsf(gLi[e])));
    auto split = [](float b) {  // b in two FP16 parts
        const __half hi = __float2half_rn(b), lo = __float2half_rn(b - __half2float(hi));
        const __half2 h2 = __halves2half2(hi, lo);
        return *reinterpret_cast<const uint32_t*>(&h2);
    };
    for (int e = tid; e < 128 * 4; e += 256) {  // W1: 128 rows x 32 K (4 x 8-element groups)
        const int r = e >> 2, kc = e & 3, gr = 128 * rank + r;
        uint4 v = bf16x8_to_f16x8(*reinterpret_cast<const uint4*>(W1 + gr * 32 + kc * 8), 1.0f);
        if (kc == 3) v.w = split(b1[gr]);  // K columns 30, 31
        *reinterpret_cast<uint4*>(res + R_W1 + canon(r, 8 * kc, 512)) = v;
    }
    {  // W4 / 2: 8 rows x 256 K
        const int r = tid >> 5, kc = tid & 31;
        *reinterpret_cast<uint4*>(res + R_W4 + canon(r, 8 * kc, 4096)) =
            bf16x8_to_f16x8(*reinterpret_cast<const uint4*>(W4 + (8 * rank + r) * 256 + kc * 8), 0.5f);
    }
    if (tid < 128)
        *reinterpret_cast<uint4*>(res + R_BB + tid * 16) =
            make_uint4(split(b2[128 * rank + tid]), split(b3[128 * rank + tid]), 0u, 0u);
    if (tid < 32) {  // per layer two core matrices: 8 rows x K 0..7, K 8..15
        const int l = tid >> 4, group = (tid >> 3) & 1, r = tid & 7;
        const uint32_t one = group == 0 ? 0x3c003c00u : 0u;
        *reinterpret_cast<uint4*>(res + R_ONES + l * ONES_BYTES + group * 128 + r * 16) =
            make_uint4(l == 0 ? one : 0u, l == 1 ? one : 0u, 0u, 0u);
    }
    __syncthreads();
    int li_exp = 0;
    frexpf(__uint_as_float(li_max), &li_exp);
    const int li_k = li_max ? max(-60, min(60, 14 - li_exp)) : 0;  // s = 2^li_k
    const float li_s = ldexpf(1.0f, li_k);
    for (int e = tid; e < 16 * 32; e += 256) {  // s L^-1 = L_hi + L_lo, rows i and K columns j, zero-padded
        const int r = e >> 5, i = 16 * rank + r, j = e & 31;
        const float v = (i < NF && j <= i) ? gLi[i * NF + j] * li_s : 0.0f;
        const __half hi = __float2half_rn(v);
        *reinterpret_cast<__half*>(res + R_LH + canon(r, j, 512)) = hi;
        *reinterpret_cast<__half*>(res + R_LL + canon(r, j, 512)) = __float2half_rn(v - __half2float(hi));
    }
    float* o = reinterpret_cast<float*>(res + R_NV);
    for (int e = tid; e < NV_BYTES / 4; e += 256) {
        float v = 0.0f;
        if (e < NV_XR) v = nv[e];
        else if (e < NV_YM) v = 1.0f / nv[e];  // (the deviations xs are kept as reciprocals)
        else if (e < NV_THR) v = nv[e];
        else if (e == NV_THR) v = nv[4 * NF + 2 * NO + NF * NF];
        else if (e == NV_S2) v = ldexpf(1.0f, -2 * li_k);
        else if (e < NV_COUNT) v = b4[e - NV_B4];
        o[e] = v;
    }
}

}  // namespace

size_t mlp_infer_stage_bytes() { return (size_t)2 * RES_BYTES; }

cudaError_t launch_mlp_infer_stage(const float* nv, const __nv_bfloat16* const W[4], const float* const b[4],
                                   uint8_t* stage, cudaStream_t s)
{
    tile_resident_kernel<<<WH_BLOCKS + 2, 256, 0, s>>>(W[0], b[0], W[1], b[1], W[2], b[2], W[3], b[3], nv, stage);
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const double* feat, int64_t n, const uint8_t* stage, double* lp6, uint8_t* in_region,
                             int* err, cudaStream_t s)
{
    static bool attr_set[64] = {};  // the attribute is per function and device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, INFER_SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    if (n <= 0) return cudaSuccess;
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t pairs = (n + 255) / 256, most = sms / 2;
    InferArgs g{};
    g.feat = feat;
    g.n = n;
    g.feat_wide = ((uintptr_t)feat & 15u) == 0;
    g.res = stage;
    g.lp6 = lp6;
    g.in_region = in_region;
    g.err = err;
    mlp_infer_kernel<<<(unsigned)(2 * (pairs < most ? pairs : most)), IT_ALL, INFER_SMEM, s>>>(g);
    return cudaGetLastError();
}

}  // namespace ptadd
