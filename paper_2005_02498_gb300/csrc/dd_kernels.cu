// dd_kernels.cu -- the pair stage of one explicit DD step on the GPU (Sec. 2.1 of
// the paper):
//   seg_prep      : per-segment source records from the current positions
//   pair_fp64 / pair_mixed : O(N^2) stress at the 4 Gauss points of every target
//                   segment, contracted with its Burgers vector, folded into
//                   the two nodal force parts of the segment (PK force, linear
//                   shape functions)
// The O(N) rest of the step (forces, velocities, Lp and rho, the Euler update, the
// next step's records) is step.cu's.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <math.h>

#include "chain.cuh"
#include "chunk_rule.cuh"
#include "pair_tile.cuh"
#include "ptadd_internal.cuh"
#include "seg_field.cuh"

namespace ptadd {

// ----------------------------------------------------------- seg_prep
__global__ void seg_prep_kernel(int64_t n, const double* __restrict__ pos, const int32_t* __restrict__ nxt,
                                const int32_t* __restrict__ loop_of, const double* __restrict__ loop_b,
                                double* __restrict__ src, float* __restrict__ src32, float* __restrict__ srcdf,
                                double ox, double oy, double oz, int origin_node0, double a2)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t j = nxt[i];
    const int k = loop_of[i];
    const double x1[3] = {pos[i], pos[n + i], pos[2 * n + i]};
    const double x2[3] = {pos[j], pos[n + j], pos[2 * n + j]};
    const double b[3] = {loop_b[3 * k], loop_b[3 * k + 1], loop_b[3 * k + 2]};
    double o[3] = {ox, oy, oz};
    if (origin_node0)
        for (int e = 0; e < 3; ++e) o[e] = rint(pos[e * n]);
    seg_records(x1, x2, b, o, a2, src + (int64_t)SRC_STRIDE * i, src32 ? src32 + (int64_t)SRC32_STRIDE * i : nullptr,
                srcdf ? srcdf + (int64_t)SRCDF_STRIDE * i : nullptr);
}

cudaError_t launch_seg_prep(const DevNetwork& net, int precision, const Consts& c, cudaStream_t st)
{
    const int64_t n = net.n_nodes;
    if (n == 0) return cudaSuccess;
    const bool mixed = precision == (int)PTADD_MIXED;
    seg_prep_kernel<<<(unsigned)((n + 63) / 64), 64, 0, st>>>(n, net.pos[net.cur], net.nxt, net.loop_of, net.loop_b,
                                                              net.src, mixed ? net.src32 : nullptr,
                                                              mixed ? nullptr : net.srcdf, net.origin[0],
                                                              net.origin[1], net.origin[2], net.origin_node0 ? 1 : 0,
                                                              c.a2);
    return cudaGetLastError();
}

// ------------------------------------------------------------ pair stage
// Grid: x = target tiles of one segment per thread (mixed: MIX_TPB, FP64: a
// warp), y = source chunks.  Each block runs one tile (pair_tile.cuh): it
// stages source records through shared memory; every thread walks them in the
// same order (broadcast reads) and accumulates (sigma b') at its 4 Gauss points.
constexpr int MIX_TPB = 32;
constexpr int MIX_MAX_CHUNKS = 64;
constexpr int MIX_TILE = 192;  // sources per tile (one plain FP32 sum), staged 32 at a time
// One-warp blocks, 16 per SM.  Bound by the FP32 pipe (177 packed instructions per
// source and warp, two cycles each, and 12 plain ones; 69 % of the active cycles, the rest being the
// latency of the formula's chain to the four warps of a scheduler); 16 warps at 128 registers (16 bytes spilled
// outside the loop's arithmetic) keep it busier than 12 at 160.  32 768 / 8192 segments:
// 13.28 / 0.947 ms per launch, blocks of two warps 13.38 / 0.948, of four 13.41 / 0.987
// (the tail is a warp's tile long, not a block's), three blocks of four warps 13.82 / 1.066.
constexpr int MIX_MINB = 16;

// FP64 path.  Bound by the FP32 pipe: 1475 packed FP32 instructions per
// source and warp, two pipe cycles each, and 33 plain ones: 3000 of the 3650 cycles that a source
// takes on a full scheduler.  32 768 segments: 96.5 ms per evaluation (1.11e10
// pairs/s), 826 ms when every pair ran on the FP64 pipe; 512 segments: 51
// against 560 us per launch.  A tile's set-up and its closing stay off the FP64
// pipe (64 cycles per warp instruction): the targets' D and b' come split from
// the records, the forces of a group are formed in double-float, and only tiles
// with near pairs (or the applied stress) run the FP64 assembly (42 segments:
// 21.0 -> 18.8 us, 1485 segments 190 -> 183).  One-warp blocks: 16 at 128 registers per thread
// run 8192 segments in 6.15 ms, 12 at 168 in 6.19, 8 in 6.35; blocks of four
// warps the same.  The points of a pair go through one copy of the code two at
// a time: with all four unrolled the loop (62 KB) missed the instruction cache
// (9.8 ms).
constexpr int DF_MINB = 16;

__global__ void __launch_bounds__(32, DF_MINB) pair_fp64_kernel(TileArgs base, int64_t n_tgt, int64_t chunk_len,
                                                                Consts c)
{
    __shared__ DFSmem sm;
    chain_wait();
    chain_next();
    TileArgs a = base;
    a.t_begin = (int64_t)blockIdx.x * 32;
    a.t_count = min((int64_t)32, n_tgt - a.t_begin);
    a.js = (int64_t)blockIdx.y * chunk_len;
    a.je = min(a.n, a.js + chunk_len);
    a.add_app = blockIdx.y == 0;
    a.fp = base.fp + (int64_t)blockIdx.y * 6 * a.n;
    pair_tile_fp64(a, c, sm);
}

__global__ void __launch_bounds__(MIX_TPB, MIX_MINB) pair_mixed_kernel(TileArgs base, int64_t n_tgt, int64_t chunk_len,
                                                             Consts c, float near2)
{
    __shared__ MixSmem<MIX_TILE, MIX_TPB> sm;
    chain_wait();
    chain_next();
    TileArgs a = base;
    a.t_begin = (int64_t)blockIdx.x * MIX_TPB;
    a.t_count = min((int64_t)MIX_TPB, n_tgt - a.t_begin);
    a.js = (int64_t)blockIdx.y * chunk_len;
    a.je = min(a.n, a.js + chunk_len);
    a.add_app = blockIdx.y == 0;
    a.fp = base.fp + (int64_t)blockIdx.y * 6 * a.n;
    pair_tile_mixed<MIX_TILE, MIX_TPB>(a, c, near2, sm);
}

// SMs and resident blocks per SM of the FP64 kernel, queried once per device.
static void pair_slots(int& sms, int& per_sm)
{
    static std::atomic<int> cached[64][2];  // [device] -> {sms, blocks per SM}; 0: not yet
    int dev = 0;
    sms = 152;
    per_sm = 16;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 &&
        cached[dev][0].load(std::memory_order_acquire) > 0) {
        sms = cached[dev][0].load(std::memory_order_relaxed);
        per_sm = cached[dev][1].load(std::memory_order_relaxed);
        return;
    }
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pair_fp64_kernel, 32, 0);
    if (per_sm < 1) per_sm = 1;
    if (dev >= 0 && dev < 64) {
        cached[dev][1].store(per_sm, std::memory_order_relaxed);
        cached[dev][0].store(sms, std::memory_order_release);
    }
}

int device_sms()
{
    int sms, per_sm;
    pair_slots(sms, per_sm);
    return sms;
}

int64_t fp64_slots()
{
    int sms, per_sm;
    pair_slots(sms, per_sm);
    return (int64_t)sms * per_sm;
}

int choose_chunks(int64_t n_tgt, int64_t n_src, int max_chunks, int precision)
{
    if (precision != (int)PTADD_MIXED) {
        int64_t len = chunk_len_rule(fp64_slots(), (n_tgt + 31) / 32, n_src);
        len = std::max(len, (n_src + max_chunks - 1) / max_chunks);
        return (int)((n_src + len - 1) / len);
    }
    // The chunk count from blocks of 128 targets (four of the kernel's one-warp blocks): 48 per SM, in
    // chunks of at least 256 sources, so that the per-block set-up and the nodal output stay small
    // next to the pair work, unless that leaves less than three per SM (a small network): then chunks
    // down to 32 sources, so that the few targets' work (and their FP64 near pairs) spreads over more SMs.
    // us a step by chunks, [the rule's]: 512 segments 160.8 in 2, 86.2 in 8, [74.4 in 16]; 2048: 164.1 in
    // 8, 139.3 in 16, 134.0 in 48, [134.7 in 64]; 4096: 361 in 8, [339 in 16], 302 in 32, 298 in 48; 8192: 984
    // in 16, [971 in 32], 954 in 64; 16 384: 3600 in 16, [3489 in 57], 3454 in 32; 32 768: 13 447 in 16,
    // [13 388 in 29], 13 358 in 48.  So about 4096 segments 32 chunks would be 11 % faster, elsewhere the rule is
    // within 2 %; but a chunk's start is where the FP32 sums start, and moving it moves averaged
    // rates by 1e-9.
    int sms, per_sm;
    pair_slots(sms, per_sm);
    const int64_t tiles_t = (n_tgt + 127) / 128;
    int64_t cap = n_src / 256;
    if (tiles_t * cap < (int64_t)sms * 3) cap = std::max<int64_t>(cap, n_src / 32);
    if (cap > MIX_MAX_CHUNKS) cap = MIX_MAX_CHUNKS;
    if (cap > max_chunks) cap = max_chunks;
    if (cap < 1) cap = 1;
    const int64_t want_blocks = (int64_t)sms * 48;
    int64_t ch = (want_blocks + tiles_t - 1) / (tiles_t > 0 ? tiles_t : 1);
    if (ch > cap) ch = cap;
    if (ch < 1) ch = 1;
    return (int)ch;
}

cudaError_t launch_pair(const DevNetwork& net, const int32_t* tgt, int64_t n_tgt, int chunks, int precision,
                        const Consts& c, const double sh[6], cudaStream_t st, bool chained)
{
    const int64_t n = net.n_nodes;
    if (n_tgt == 0 || n == 0) return cudaSuccess;
    const int64_t chunk_len = (n + chunks - 1) / chunks;
    TileArgs a{};
    a.pos = net.pos[net.cur];
    a.n = n;
    a.nxt = net.nxt;
    a.src = net.src;
    a.src32 = net.src32;
    a.srcdf = net.srcdf;
    a.tgt = tgt;
    for (int k = 0; k < 6; ++k) a.sh[k] = sh[k];
    for (int k = 0; k < 3; ++k) a.origin[k] = net.origin[k];
    a.fp = net.fpart;
    a.fp_stride = n;
    a.node_base = 0;
    a.near_count = net.near_count;
    a.k64 = net.k64;
    if (precision == (int)PTADD_MIXED) {
        dim3 grid((unsigned)((n_tgt + MIX_TPB - 1) / MIX_TPB), (unsigned)chunks);
        const float near2 = (float)((NEAR_FACTOR * NEAR_FACTOR + 1.0) * c.a2);
        if (chained) return launch_chained(pair_mixed_kernel, grid, MIX_TPB, 0, st, a, n_tgt, chunk_len, c, near2);
        pair_mixed_kernel<<<grid, MIX_TPB, 0, st>>>(a, n_tgt, chunk_len, c, near2);
        return cudaGetLastError();
    }
    const dim3 grid((unsigned)((n_tgt + 31) / 32), (unsigned)chunks);
    if (chained) return launch_chained(pair_fp64_kernel, grid, 32, 0, st, a, n_tgt, chunk_len, c);
    pair_fp64_kernel<<<grid, 32, 0, st>>>(a, n_tgt, chunk_len, c);
    return cudaGetLastError();
}

}  // namespace ptadd
