// sde_denoise.cu -- tensor-core (tcgen05) kernels of the learned dose denoiser.
//
// The denoiser is a 3D convolutional encoder-decoder applied to a low-history dose
// and the density map; its convolutions are implicit GEMMs on the 5th-generation
// tensor core with BF16 operands in shared memory and FP32 accumulators in tensor
// memory.  This file holds the GEMM building block and its C entry point.
#include <cuda_bf16.h>
#include <stdio.h>

#include <algorithm>
#include <mutex>

#include "sde_dose.h"
#include "sde_tables.h"
#include "sde_denoise.h"
#include "sde_umma.cuh"

namespace sde {

namespace {

constexpr long long kWaitCycles = 1ll << 31;  // ~1 s at 2 GHz: a stuck wait sets the error flag

// D[M x N] (FP32, row-major) = A[M x K] x B[N x K]^T with A, B row-major BF16 (both
// K-major).  One CTA of 128 threads per 128-row tile of D; K is staged in chunks of
// 64 through shared memory in the core-matrix layout; one thread issues the MMAs.
__global__ void __launch_bounds__(128) k_gemm_bf16(const __nv_bfloat16* __restrict__ A,
                                                   const __nv_bfloat16* __restrict__ B, float* __restrict__ D,
                                                   int M, int N, int K, unsigned int* status) {
    constexpr int KC = 64;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;
    unsigned char* sB = smem + 128 * KC * 2;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sB + 256 * KC * 2);
    uint32_t* slot = reinterpret_cast<uint32_t*>(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * 128;
    const uint32_t ncols = N <= 32 ? 32u : N <= 64 ? 64u : N <= 128 ? 128u : 256u;
    if (warp == 0) {
        umma::tmem_alloc(slot, ncols);
        umma::tmem_relinquish();
    }
    if (tid == 0) umma::mbar_init(mbar, 1);
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tbase = *slot;
    const uint32_t idesc = umma::idesc_bf16_f32(128, N);
    bool ok = true;
    int it = 0;
    for (int k0 = 0; k0 < K; k0 += KC, ++it) {
        const int kc = min(KC, K - k0);
        const int q8 = kc >> 3;
        for (int c = tid; c < 128 * q8; c += 128) {
            int r = c / q8, q = c - r * q8;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (m0 + r < M) v = *reinterpret_cast<const uint4*>(A + (size_t)(m0 + r) * K + k0 + q * 8);
            *reinterpret_cast<uint4*>(sA + umma::core_offset(r, q * 8, kc)) = v;
        }
        for (int c = tid; c < N * q8; c += 128) {
            int r = c / q8, q = c - r * q8;
            uint4 v = *reinterpret_cast<const uint4*>(B + (size_t)r * K + k0 + q * 8);
            *reinterpret_cast<uint4*>(sB + umma::core_offset(r, q * 8, kc)) = v;
        }
        umma::fence_async_smem();
        umma::fence_before_sync();
        __syncthreads();
        umma::fence_after_sync();
        if (tid == 0) {
            for (int ks = 0; ks < (kc >> 4); ++ks) {
                uint64_t ad = umma::smem_desc(umma::smem_addr(sA) + ks * 256, 128, 16 * kc);
                uint64_t bd = umma::smem_desc(umma::smem_addr(sB) + ks * 256, 128, 16 * kc);
                umma::mma_bf16(tbase, ad, bd, idesc, (k0 > 0 || ks > 0) ? 1u : 0u);
            }
            umma::mma_commit(mbar);
        }
        bool done = umma::mbar_wait(mbar, (uint32_t)(it & 1), kWaitCycles);
        umma::fence_after_sync();
        if (!__syncthreads_and(done ? 1 : 0)) {
            ok = false;
            break;
        }
    }
    if (ok) {
        for (int c = 0; c < N; c += 8) {
            float v[8];
            umma::tmem_ld8(tbase + ((uint32_t)(32 * warp) << 16) + (uint32_t)c, v);
            int row = m0 + 32 * warp + lane;
            if (row < M)
                for (int j = 0; j < 8; ++j) D[(size_t)row * N + c + j] = v[j];
        }
    } else if (tid == 0) {
        atomicOr(status, 1u);
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    if (warp == 0) umma::tmem_dealloc(tbase, ncols);
}

std::mutex g_status_mutex;
unsigned int* g_status[64] = {};

// A device status word per device (allocated on first use).
cudaError_t status_word(unsigned int** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_status_mutex);
    if (!g_status[dev]) {
        e = cudaMalloc(&g_status[dev], sizeof(unsigned int));
        if (e != cudaSuccess) return e;
        e = cudaMemset(g_status[dev], 0, sizeof(unsigned int));
        if (e != cudaSuccess) return e;
    }
    *out = g_status[dev];
    return cudaSuccess;
}

// Stream-ordered scratch memory from a pool of the library's own, one per device.  The device's
// default pool gives its memory back at every wait, so a call after one mapped its few hundred
// kilobytes anew (a convolution and a wait: 375 us against 155 back to back); this pool keeps up to
// 32 MB between waits and gives them back when a denoiser is destroyed.  While the stream
// is being captured the allocation becomes a node of the graph as before.  The error that is cleared is
// of this library's own CUDA runtime (linked statically: a caller's pending errors are kept by the
// caller's) and of a query here, or of an earlier call, which has returned it.
constexpr uint64_t kScratchKept = 32ull << 20;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[64] = {};

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    int dev = -1;
    cudaMemPool_t pool = nullptr;
    if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone &&
        cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lock(g_pool_mutex);
        if (!g_pool[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            uint64_t kept = kScratchKept;
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // another thread may be capturing
            cudaThreadExchangeStreamCaptureMode(&mode);
            if (cudaMemPoolCreate(&g_pool[dev], &props) != cudaSuccess)
                g_pool[dev] = nullptr;
            else
                cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &kept);
            cudaThreadExchangeStreamCaptureMode(&mode);
        }
        pool = g_pool[dev];
    }
    cudaGetLastError();
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, st) : cudaMallocAsync(p, bytes, st);
}

int report(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return SDE_OK;
    char m[256];
    snprintf(m, sizeof m, "%s: %s", what, cudaGetErrorString(e));
    set_last_error(m);
    return e == cudaErrorMemoryAllocation ? SDE_ENOMEM : SDE_ECUDA;
}

}  // namespace

cudaError_t denoise_status_word(unsigned int** out) { return status_word(out); }

void denoise_scratch_trim() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (g_pool[dev]) cudaMemPoolTrimTo(g_pool[dev], 0);
}

// Reads and clears the device status word; SDE_EDEVICE when a tensor-core wait timed out.
int denoise_check_status(cudaStream_t st) {
    unsigned int* d_status = nullptr;
    int rc = report(status_word(&d_status), "status word");
    if (rc) return rc;
    unsigned int h = 0;
    rc = report(cudaMemcpyAsync(&h, d_status, sizeof h, cudaMemcpyDeviceToHost, st), "status copy");
    if (rc) return rc;
    rc = report(cudaStreamSynchronize(st), "status sync");
    if (rc) return rc;
    if (h) {
        cudaMemsetAsync(d_status, 0, sizeof h, st);
        cudaStreamSynchronize(st);
        set_last_error("a tensor-core completion wait timed out (result not written)");
        return SDE_EDEVICE;
    }
    return SDE_OK;
}

}  // namespace sde

using namespace sde;

extern "C" int sde_gemm_bf16(const void* d_A, const void* d_B, float* d_D, int M, int N, int K, void* stream) {
    if (!d_A || !d_B || !d_D || M < 1 || N < 16 || N > 256 || (N % 16) || K < 16 || (K % 16)) {
        set_last_error("sde_gemm_bf16: need M >= 1, N a multiple of 16 in [16, 256], K a multiple of 16");
        return SDE_EINVAL;
    }
    if (((uintptr_t)d_A | (uintptr_t)d_B) & 15) {
        set_last_error("sde_gemm_bf16: A and B must be 16-byte aligned");
        return SDE_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    unsigned int* d_status = nullptr;
    int rc = report(status_word(&d_status), "status word");
    if (rc) return rc;
    const size_t smem = 128 * 64 * 2 + 256 * 64 * 2 + 64;
    rc = report(cudaFuncSetAttribute(k_gemm_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                "cudaFuncSetAttribute");
    if (rc) return rc;
    k_gemm_bf16<<<(M + 127) / 128, 128, smem, st>>>(static_cast<const __nv_bfloat16*>(d_A),
                                                       static_cast<const __nv_bfloat16*>(d_B), d_D, M, N, K,
                                                       d_status);
    rc = report(cudaGetLastError(), "k_gemm_bf16 launch");
    if (rc) return rc;
    return denoise_check_status(st);
}

// ============================================================================
// 3D convolution (3x3x3, stride 1, zero padding 1) as implicit GEMMs on the tensor
// core.  Activations are channels-last BF16: x[n][z][y][x][c].  Weights w[co][tap][ci]
// (tap = 9 kz + 3 ky + kx).
// ============================================================================
namespace sde {
namespace {

// ----------------------------------------------------------------------------
// Brick convolution.  A work item computes Ty full output rows (all x) of one z plane
// for Cp output channels.  Per 16-channel chunk of Cin the zero-padded input "brick" --
// planes z-1..z+1, rows y0-1..y0+Ty, columns -1..W -- is staged in shared memory once,
// as two 8-channel planes in which brick position f = (zb Yb + yb) P + xp (P = W + 2,
// Yb = Ty + 2) holds 16 bytes.  In that layout 8 consecutive positions form a K-major
// core matrix, so the A operand of tap (dz, dy, dx) for an M tile starting at brick
// position f0 is the same buffer read from f0 + (dz Yb + dy) P + dx: the 27 taps are 27
// descriptor offsets, not 27 copies.  The input is padded channel-group-major, so each
// (channel group, plane) part of the brick is one contiguous run of Yb P x 16 bytes in
// global memory and a chunk arrives in six bulk copies.  When W is a multiple of 128 an M
// tile is 128 consecutive x of one output row and no padding column is computed;
// otherwise M tiles of 128 consecutive positions cover the Ty rows including their
// padding columns and the epilogue drops the rows that are not output voxels.
//
// Persistent and warp-specialised: one thread in each of three copy warps, one per plane of the
// brick, streams that plane's runs and weights into a ring of shared-memory stages (a "full"
// barrier per stage and plane completes when the bytes of its copies have landed); two MMA
// warps issue tcgen05.mma for the M tiles of their parity, plane by plane, into one of two
// tensor-memory accumulators, and release planes and accumulators through tcgen05.commit; the
// epilogue groups turn a finished tile into output (bias, leaky ReLU, BF16 or FP32 store) while the
// tensor core works on the next ones.  Every wait is bounded; a timeout sets a shared abort flag
// that ends all roles' loops, and each copy thread waits for its copies in flight before the CTA
// exits.
//
// The copy and MMA roles run one warp each, at some seven cycles an instruction, so their loops
// hold no index division, no dispatch and no address that a step could carry: with those a plane
// took them 500 cycles whatever its MMAs (100 to 500).  The stages are released a plane at a time,
// which with two of them keeps five of six planes in flight.  192x128x128: 16 -> 32 channels 150 ->
// 117 us, 32 -> 32 200 -> 165 (145 with the epilogue's 16-column blocks below; the folded epilogue
// bounds it: 110 without), 96 -> 32 472 -> 336 (operand reads and copies share the shared memory's
// port), inference 1.89 -> 1.55 ms (1.46 with those blocks).
// ----------------------------------------------------------------------------
constexpr int kPipeStages = 2;
constexpr int kPipeHeader = 1024;  // barriers, tensor-memory slot, abort flag

// One try first: the clock and the abort flag cost a role that runs alone in its warp more than
// the wait when the phase is over already.
__device__ __forceinline__ bool pipe_wait(uint64_t* m, uint32_t parity, volatile int* abort_flag) {
    if (umma::mbar_try_wait(m, parity)) return true;
    const long long t0 = clock64();
    while (!umma::mbar_try_wait_long(m, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// Epilogue warps of the brick convolution, groups of four that cover a tile's 128 lanes (warp &
// 3: the tensor-memory lane quarter); the two MMA warps and the copy warps follow them.
constexpr int kConvGroups = 4;
constexpr int kConvWorkers = 4 * kConvGroups;
constexpr int kConvCopyWarps = 3;  // one per brick plane
constexpr int kConvThreads = 32 * (kConvWorkers + 2 + kConvCopyWarps);

// AND of a predicate over the NT worker threads of a kernel (its warps 0 .. NT/32 - 1),
// named barrier 1.
template <int NT>
__device__ __forceinline__ bool workers_all(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\tsetp.ne.u32 pi, %1, 0;\n\tbar.red.and.pred po, 1, %2, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(NT)
        : "memory");
    return r != 0;
}

// Brick position of output row 0's first M-tile row, shifted to tile m (tap offsets are
// added to it): row tiles are 128 x of one output row, flat tiles 128 consecutive positions
// starting at output (y0, x = -1).
__device__ __forceinline__ int tile_base(int m, bool rowtile, int P, int Yb, int tpr) {
    return rowtile ? (Yb + 1) * P + 1 + (m / tpr) * P + (m % tpr) * 128 : (Yb + 1) * P + 128 * m;
}

// What an MMA warp needs beside the plan: barriers, the first stage's operand descriptors (A at
// the plane z - 1 of tap (-1, -1, -1)'s row offset 0, B at tap 0) and the resident weights'.
struct IssueArgs {
    uint64_t *full, *empty, *tfull, *tempty;
    volatile int* abort_flag;
    uint64_t a0, b0;
    uint32_t tbase, idesc, leader;
    int items, nchunk, Cp, tpr;
};

// The MMA warp of the M tiles of parity PAR: per item, chunk and plane dz the taps' MMAs in order,
// straight through with an add or two per instruction.  A warp issues alone, at some seven
// cycles an instruction, and a plane is 3 to 9 MMAs per tile: a dispatch on the tile count and
// descriptors formed per plane took as long as the MMAs (500 cycles a plane).
//  - unfolded: nine taps per plane, A's start field the plane's plus tile base and tap offset, B's a
//    tap tile (Cp x 16 BF16 = 2 Cp units of 16 bytes) further each;
//  - folded (one 128-voxel row per tile): per (z, y) tap pair one MMA of N = 3 Cp whose B is the
//    three consecutive x-tap tiles of the pair and whose A is the pair's dx = 0 window;
//    accumulator column block j then holds the window's product with the dx = j - 1 weights,
//    and the epilogue adds the blocks shifted by one position.
// The start fields stay within 14 bits (shared addresses below 256 KB, lowest start one position
// into the stage), so adding to the low word never carries or borrows into the others.
template <bool FOLD, int TILES, int PAR>
__device__ __forceinline__ void conv_issue(const BrickPlan& b, const IssueArgs& g) {
    static_assert(kPipeStages == 2, "stages alternate");
    const uint32_t a_hi = (uint32_t)(g.a0 >> 32), b_hi = (uint32_t)(g.b0 >> 32);
    const int P = b.P, plane = b.Yb * P, Cp = g.Cp, acc_cols = TILES * Cp * (FOLD ? 3 : 1);
    uint32_t tb[TILES], td[TILES];
#pragma unroll
    for (int m = PAR; m < TILES; m += 2) {
        tb[m] = (uint32_t)g.a0 + (uint32_t)(tile_base(m, b.rowtile != 0, P, b.Yb, g.tpr) - plane - P);
        td[m] = (uint32_t)(m * Cp * (FOLD ? 3 : 1));
    }
    const uint32_t stage = (uint32_t)b.stage >> 4, w_chunk = (uint32_t)(27 * 2 * Cp);
    uint32_t soff = 0, par = 0, acc_par = 1;
    int acc = 0;
    bool ok = true;
    for (int j = 0; j < g.items; ++j) {
        if (j >= b.nacc) ok = pipe_wait(&g.tempty[acc], acc_par, g.abort_flag);
        const uint32_t dacc = g.tbase + (uint32_t)(acc * acc_cols);
        for (int c = 0; c < g.nchunk; ++c) {
            uint64_t* const full = g.full + (soff ? 3 : 0);
            uint64_t* const empty = g.empty + (soff ? 3 : 0);
            const uint32_t bs = (uint32_t)g.b0 + (b.wres ? (uint32_t)c * w_chunk : soff);
#pragma unroll
            for (int dz = 0; dz < 3; ++dz) {
                ok = ok && pipe_wait(&full[dz], par, g.abort_flag);
                if (!__all_sync(0xffffffffu, ok)) return;
                umma::fence_after_sync();
                const uint32_t as = soff + (uint32_t)(dz * plane), bz = bs + (uint32_t)(18 * Cp * dz);
                const uint32_t first = dz > 0 || c > 0 ? 1u : 0u;
#pragma unroll
                for (int q = 0; q < (FOLD ? 3 : 9); ++q) {
                    // folded: the middle x offset of row pair q and its three tap tiles
                    const uint32_t ao = as + (uint32_t)((FOLD ? q : q / 3) * P + (FOLD ? 0 : q % 3 - 1));
                    const uint32_t bo = bz + (uint32_t)((FOLD ? 6 : 2) * Cp * q);
#pragma unroll
                    for (int m = PAR; m < TILES; m += 2)
                        umma::mma_bf16_warp(g.leader, dacc + td[m], tb[m] + ao, a_hi, bo, b_hi, g.idesc, q > 0 ? 1u : first);
                }
                umma::mma_commit_warp(g.leader, &empty[dz]);
            }
            par ^= soff ? 1u : 0u;
            soff = soff ? 0u : stage;
        }
        umma::mma_commit_warp(g.leader, &g.tfull[acc]);
        if (++acc == b.nacc) {
            acc = 0;
            acc_par ^= 1u;
        }
    }
}

// Named barrier over the 128 threads of one group of four epilogue warps.
__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

// Work item of the brick convolution: (sample, Cout part, row block, z plane), z fastest.  A CTA
// takes every gridDim.x-th one and steps by increments (its roles run one thread a warp, where an
// integer division costs a hundred cycles).
struct BrickItems {
    int left;             // items still to come, this one included
    int z, yb, part, n;
    int sz, syb;          // step in (row block, z plane)
    __device__ __forceinline__ BrickItems(const BrickPlan& b, int D) {
        int item = blockIdx.x;
        const int G = gridDim.x;
        left = (b.items - item + G - 1) / G;
        sz = G % D;
        syb = G / D;
        z = item % D;
        item /= D;
        yb = item % b.nyb;
        item /= b.nyb;
        part = item % b.nsplit;
        n = item / b.nsplit;
    }
    __device__ __forceinline__ void next(const BrickPlan& b, int D) {
        --left;
        z += sz;
        yb += syb;
        if (z >= D) {
            z -= D;
            ++yb;
        }
        for (; yb >= b.nyb; yb -= b.nyb)
            if (++part == b.nsplit) {
                part = 0;
                ++n;
            }
    }
};

// Sixteen accumulator columns of this lane's row of a tile, from tcol on, as packed pairs.
// Folded: out[x] = D[x-1][co] + D[x][Cp + co] + D[x+1][2 Cp + co]; x - 1 and x + 1 of a lane
// quarter's edge lanes belong to the neighbouring quarter (another warp of the group), x = -1 and
// x = 128 are padding (their D is zero).  Edge lanes publish their columns in xch
// ([2][quarter][16]), all warps of the group meet, and the edge lanes add what their
// neighbours published.
template <bool FOLD>
__device__ __forceinline__ void tile_columns(uint32_t tcol, int Cp, float* xch, bool one_buffer, int quarter, int lane,
                                             int barrier, float2 (&out)[8]) {
    uint32_t v[16];
    if (FOLD) {
        uint32_t lo[16], hi[16];
        umma::tmem_ld16_nowait(tcol, lo);
        umma::tmem_ld16_nowait(tcol + (uint32_t)(2 * Cp), hi);
        umma::tmem_wait_ld16(lo);
        umma::tmem_touch16(hi);
        if (lane == 31 || lane == 0) {
            uint4* dst = reinterpret_cast<uint4*>(xch + (lane == 31 ? 0 : 64) + quarter * 16);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                dst[q] = lane == 31 ? make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3])
                                    : make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
        }
        umma::tmem_ld16_nowait(tcol + (uint32_t)Cp, v);
        const uint32_t ml = lane == 0 ? 0u : ~0u, mr = lane == 31 ? 0u : ~0u;
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
            float2 l, r;
            l.x = __uint_as_float(__shfl_up_sync(0xffffffffu, lo[e], 1) & ml);
            l.y = __uint_as_float(__shfl_up_sync(0xffffffffu, lo[e + 1], 1) & ml);
            r.x = __uint_as_float(__shfl_down_sync(0xffffffffu, hi[e], 1) & mr);
            r.y = __uint_as_float(__shfl_down_sync(0xffffffffu, hi[e + 1], 1) & mr);
            out[e / 2] = __fadd2_rn(l, r);
        }
        group_sync(barrier);
        const bool left = lane == 0;
        if ((left && quarter > 0) || (lane == 31 && quarter < 3)) {
            const float4* src = reinterpret_cast<const float4*>(xch + (left ? (quarter - 1) * 16 : 64 + (quarter + 1) * 16));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = src[q];
                out[2 * q] = __fadd2_rn(make_float2(w.x, w.y), out[2 * q]);
                out[2 * q + 1] = __fadd2_rn(make_float2(w.z, w.w), out[2 * q + 1]);
            }
        }
        __syncwarp();
        if (one_buffer) group_sync(barrier);  // the next columns go to the same buffer
    } else {
        umma::tmem_ld16_nowait(tcol, v);
    }
    umma::tmem_wait_ld16(v);
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        const float2 d = make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
        out[e / 2] = FOLD ? __fadd2_rn(d, out[e / 2]) : d;
    }
}

// Where a lane writes sixteen channels: the 16-byte unit of its voxel in the first of the two
// channel groups of y (FP32 output: its voxel index), that of its first child on the doubled
// grid, and whether it is an output voxel.
struct TileVoxel {
    size_t at, up, mask;  // mask: as at, in the mask's tensor
    bool valid;
};

// What the epilogue does beside bias, leaky ReLU and store: nothing, the upsampled copy, or the
// adjoint of a leaky ReLU.  Kernels of their own: the code of the others cost the plain one 1 %.
enum { kConvPlain, kConvUp, kConvMask };

// Bias, leaky ReLU and the stores of the sixteen channels from ch on (tile_columns in r).
template <int MODE>
__device__ __forceinline__ void store_columns(const ConvArgs& a, const TileVoxel& t, int ch, int lane, size_t vp,
                                              float2 (&r)[8]) {
    if (a.bias) {
        const float4* bq = reinterpret_cast<const float4*>(a.bias + ch);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 w = __ldg(bq + q);
            r[2 * q] = __fadd2_rn(r[2 * q], make_float2(w.x, w.y));
            r[2 * q + 1] = __fadd2_rn(r[2 * q + 1], make_float2(w.z, w.w));
        }
    }
    if (a.relu) {
        const float2 slope = make_float2(a.slope, a.slope);
        if (a.slope > 0.f) {  // 0 < slope < 1: the larger of x and slope x
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float2 s = __fmul2_rn(slope, r[e]);
                r[e] = make_float2(fmaxf(r[e].x, s.x), fmaxf(r[e].y, s.y));
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float2 s = __fmul2_rn(slope, r[e]);
                r[e].x = r[e].x > 0.f ? r[e].x : s.x;
                r[e].y = r[e].y > 0.f ? r[e].y : s.y;
            }
        }
    }
    if (a.y_fp32) {
        if (!t.valid) return;
        if (a.y_keep) {  // leading channels only
            if (ch == 0)
#pragma unroll
                for (int e = 0; e < 8; ++e) {  // constant indices keep r in registers
                    if (2 * e < a.y_keep) static_cast<float*>(a.y)[t.at * a.y_keep + 2 * e] = r[e].x;
                    if (2 * e + 1 < a.y_keep) static_cast<float*>(a.y)[t.at * a.y_keep + 2 * e + 1] = r[e].y;
                }
        } else {
            float4* yo = reinterpret_cast<float4*>(static_cast<float*>(a.y) + t.at * a.y_cstride + a.y_coffset + ch);
#pragma unroll
            for (int q = 0; q < 4; ++q) yo[q] = make_float4(r[2 * q].x, r[2 * q].y, r[2 * q + 1].x, r[2 * q + 1].y);
        }
        return;
    }
    uint4* yo = static_cast<uint4*>(a.y) + t.at;
    uint4 val[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        __nv_bfloat162 pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pk[e] = __float22bfloat162_rn(r[4 * q + e]);
        if (MODE == kConvMask && t.valid) {  // the value rounded to BF16 first, as a pass of its own would read it
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(a.mask) + t.mask + q * vp);
            const __nv_bfloat162* y = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 m = __bfloat1622float2(y[e]);
                float2 f = __bfloat1622float2(pk[e]);
                f.x = m.x > 0.f ? f.x : f.x * a.mask_slope;
                f.y = m.y > 0.f ? f.y : f.y * a.mask_slope;
                pk[e] = __float22bfloat162_rn(f);
            }
        }
        val[q] = *reinterpret_cast<uint4*>(pk);
        if (t.valid) yo[q * vp] = val[q];
    }
    if (MODE == kConvUp) {
        // The eight children on the doubled grid.  Lane i stores child i & 1 of lane i / 2 (then of lane
        // 16 + i / 2), so that a warp's store covers whole 32-byte sectors: every lane storing its own
        // children left half of each sector to another instruction.
        const size_t row = 2 * (size_t)a.W + 2, plane = row * (2 * a.H + 2), vp_up = plane * (2 * a.D + 2);
        uint4* yu = static_cast<uint4*>(a.y_up);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int from = 16 * h + (lane >> 1);
            const size_t at = (size_t)__shfl_sync(0xffffffffu, (unsigned long long)t.up, from) + (lane & 1);
            const bool ok = __shfl_sync(0xffffffffu, (int)t.valid, from) != 0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint4 w;
                w.x = __shfl_sync(0xffffffffu, val[q].x, from);
                w.y = __shfl_sync(0xffffffffu, val[q].y, from);
                w.z = __shfl_sync(0xffffffffu, val[q].z, from);
                w.w = __shfl_sync(0xffffffffu, val[q].w, from);
                if (ok) {
                    uint4* d = yu + at + q * vp_up;
                    d[0] = w;
                    d[row] = w;
                    d[plane] = w;
                    d[plane + row] = w;
                }
            }
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(kConvThreads, 1) k_conv3d_brick(ConvArgs a, BrickPlan b) {
    extern __shared__ __align__(1024) unsigned char smem[];
    // warp-uniform for the compiler too, so that the MMA warps' operands are
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int Cin = a.Cin, Cp = b.Cp, W = a.W, H = a.H, D = a.D;
    const int P = b.P, Yb = b.Yb;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);  // [kPipeStages][3 planes]
    uint64_t* empty = full + 3 * kPipeStages;             // [kPipeStages][3 planes]
    uint64_t* tfull = empty + 3 * kPipeStages;            // [2]
    uint64_t* tempty = tfull + 2;                         // [2]
    uint64_t* wfull = tempty + 2;                         // resident weights landed
    uint32_t* slot = reinterpret_cast<uint32_t*>(smem + 160);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 164);
    const uint32_t s_stage0 = umma::smem_addr(smem) + kPipeHeader;
    if (warp == 0) {
        umma::tmem_alloc(slot, (uint32_t)b.tcols);
        umma::tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < 3 * kPipeStages; ++s) {
            umma::mbar_init(&full[s], 1);
            umma::mbar_init(&empty[s], 2);  // one commit per MMA warp
        }
        for (int s = 0; s < 2; ++s) {
            umma::mbar_init(&tfull[s], 2);
            umma::mbar_init(&tempty[s], 4 * b.tiles * (Cp >> 4));  // one arrival per warp and block of columns
        }
        umma::mbar_init(wfull, 1);
        *abort_flag = 0;
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tbase = __shfl_sync(0xffffffffu, *slot, 0);
    const int nchunk = Cin >> 4;
    const int acc_cols = b.tiles * Cp * (b.fold ? 3 : 1);
    const int tpr = W >> 7;                          // row tiles: M tiles per output row
    const uint32_t w_chunk = (uint32_t)(27 * Cp * 32);  // bytes of one chunk's weights
    const uint32_t s_wres = s_stage0 + (uint32_t)(kPipeStages * b.stage);
    const Pcg pg{D, H, W};
    BrickItems t(b, D);

    if (warp >= kConvWorkers + 2) {
        // copy warp of plane z - 1 + zb: its run of either channel group, its nine taps' weights
        const int zb = warp - kConvWorkers - 2;
        if (lane == 0) {
            const size_t row = (size_t)P * 16, plane = (size_t)(H + 2) * row, group = pg.vp() * 16;
            const unsigned char* src = reinterpret_cast<const unsigned char*>(a.x) + zb * plane;
            const unsigned char* wsrc = reinterpret_cast<const unsigned char*>(a.wpk) + zb * (w_chunk / 3);
            const uint32_t dst = s_stage0 + 128u + (uint32_t)(zb * Yb * P * 16);
            const uint32_t wdst = s_stage0 + (uint32_t)b.w_off + (uint32_t)zb * (w_chunk / 3);
            int k = 0, s = 0;
            uint32_t par = 1;  // of the "empty" phase to wait for
            if (b.wres && zb == 0) {
                umma::mbar_arrive_expect_tx(wfull, (uint32_t)nchunk * w_chunk);
                umma::bulk_g2s(s_wres, a.wpk, (uint32_t)nchunk * w_chunk, wfull);
            }
            bool ok = true;
            for (; ok && t.left > 0; t.next(b, D)) {
                const int y0 = t.yb * b.Ty;
                // padded rows y0 .. y0+Yb-1 of the plane, fewer in a last row block that passes H (the
                // rows it leaves stale feed only outputs y >= H, which the epilogue drops)
                const uint32_t run = (uint32_t)((Yb < H + 2 - y0 ? Yb : H + 2 - y0) * P * 16);
                const unsigned char* xs = src + ((size_t)t.n * (Cin >> 3) * group + (size_t)t.z * plane + (size_t)y0 * row);
                const unsigned char* ws = wsrc + (size_t)t.part * nchunk * w_chunk;
                for (int c = 0; c < nchunk; ++c, ++k) {
                    uint64_t* f = &full[3 * s + zb];
                    if (k >= kPipeStages && !(ok = pipe_wait(&empty[3 * s + zb], par, abort_flag))) break;
                    const uint32_t st = (uint32_t)(s * b.stage);
                    umma::mbar_arrive_expect_tx(f, 2u * run + (b.wres ? 0u : w_chunk / 3));
                    umma::bulk_g2s(dst + st, xs, run, f);
                    umma::bulk_g2s(dst + st + (uint32_t)b.plane, xs + group, run, f);
                    if (!b.wres) umma::bulk_g2s(wdst + st, ws, w_chunk / 3, f);
                    xs += 2 * group;
                    ws += w_chunk;
                    if (++s == kPipeStages) {
                        s = 0;
                        par ^= 1u;
                    }
                }
            }
            // no copy may still be writing shared memory when the CTA exits: wait for this thread's last
            // kPipeStages (earlier ones were consumed before their stage was reused)
            for (int kk = k > kPipeStages ? k - kPipeStages : 0; kk < k; ++kk)
                umma::mbar_wait(&full[3 * (kk % kPipeStages) + zb], (uint32_t)(kk / kPipeStages) & 1u, kWaitCycles);
            if (b.wres && zb == 0) umma::mbar_wait(wfull, 0u, kWaitCycles);
        }
        __syncwarp();
    } else if (warp >= kConvWorkers) {
        // two MMA warps (one thread can issue a tcgen05.mma only every ~65 cycles, two are
        // bound by the operand reads from shared memory): issuer iss takes the M tiles of its
        // parity, so each accumulator column range has one issuer
        const int iss = warp - kConvWorkers;
        IssueArgs g;
        g.full = full;
        g.empty = empty;
        g.tfull = tfull;
        g.tempty = tempty;
        g.abort_flag = abort_flag;
        g.a0 = umma::smem_desc(s_stage0 + 128u, (uint32_t)b.plane, 128);
        g.b0 = umma::smem_desc(b.wres ? s_wres : s_stage0 + (uint32_t)b.w_off, 128, 256);
        g.tbase = tbase;
        g.idesc = umma::idesc_bf16_f32(128, b.fold ? 3 * Cp : Cp);
        g.leader = umma::elect_one();
        g.items = t.left;
        g.nchunk = nchunk;
        g.Cp = Cp;
        g.tpr = tpr;
        if (__all_sync(0xffffffffu, !b.wres || pipe_wait(wfull, 0u, abort_flag))) {
            switch (b.tiles + (b.fold ? 100 : 0)) {
#define SDE_CONV_ISSUE(F, T)                        \
    case (F ? 100 : 0) + T:                         \
        if (iss) conv_issue<F, T, 1>(b, g);         \
        else conv_issue<F, T, 0>(b, g);             \
        break;
                SDE_CONV_ISSUE(true, 1)
                SDE_CONV_ISSUE(true, 2)
                SDE_CONV_ISSUE(true, 3)
                SDE_CONV_ISSUE(true, 4)
                SDE_CONV_ISSUE(false, 1)
                SDE_CONV_ISSUE(false, 2)
                SDE_CONV_ISSUE(false, 3)
                SDE_CONV_ISSUE(false, 4)
                SDE_CONV_ISSUE(false, 5)
                SDE_CONV_ISSUE(false, 6)
                SDE_CONV_ISSUE(false, 7)
                SDE_CONV_ISSUE(false, 8)
#undef SDE_CONV_ISSUE
                default:  // the plan keeps items to <= 8 tiles, folded ones to <= 4
                    *abort_flag = 1;
            }
        }
        __syncwarp();
    } else {
        // epilogue: the blocks of sixteen columns of the CTA's M tiles, all items' in order, go round
        // the groups.  Each warp waits for its tile's accumulator by itself; after a timeout it goes on
        // through its blocks without storing, so that the group's barriers still meet.  A group does not
        // wait for an item that it has no block of, and a wait tells an accumulator's fillings apart
        // by their parity only: with one block an item and four groups, the next item of a group is its
        // accumulator's next but one, whose wait would end at once.  So only as many groups take part as
        // have a block of every nacc-th item (b.groups).
        const int quarter = warp & 3;  // tensor-memory lanes 32 quarter .. + 31
        const int grp = warp >> 2, blocks = Cp >> 4;
        const size_t vp = pg.vp();
        const int Gy = a.y_cstride >> 3;
        // fold: per group two buffers (used in turn; one where Cp = 16 leaves room for no more) of
        // [2][lane quarter][16] values at the quarters' edges: D[x = 32 quarter + 31][co] and
        // D[x = 32 quarter][2 Cp + co]
        const bool one_buffer = Cp < 32;
        float* xbuf = reinterpret_cast<float*>(smem + b.xch) + grp * (one_buffer ? 128 : 256);
        int par = 0;
        bool ok = true;
        uint32_t acc_par = 0;
        int acc = 0, m = 0, blk = grp;
        while (grp < b.groups && t.left > 0) {
            if (blk >= blocks) {  // on to the next tile
                blk -= blocks;
                if (++m < b.tiles) continue;
                m = 0;
                t.next(b, D);
                if (++acc == b.nacc) {
                    acc = 0;
                    acc_par ^= 1u;
                }
                continue;
            }
            if (lane == 0) ok = ok && pipe_wait(&tfull[acc], acc_par, abort_flag);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            umma::fence_after_sync();
            const int c = 16 * blk, ch = t.part * Cp + c;
            const uint32_t tcol = tbase + ((uint32_t)(32 * quarter) << 16) +
                                  (uint32_t)(acc * acc_cols + m * Cp * (b.fold ? 3 : 1) + c);
            float2 r[8];
            __syncwarp();
            if (b.fold)
                tile_columns<true>(tcol, Cp, xbuf + 128 * par, one_buffer, quarter, lane, 1 + grp, r);
            else
                tile_columns<false>(tcol, Cp, nullptr, false, quarter, lane, 0, r);
            if (!one_buffer) par ^= 1;
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&tempty[acc]);  // the columns are in registers
            const int y0 = t.yb * b.Ty;
            int yy, xx;
            bool valid;
            if (b.rowtile) {
                yy = y0 + (tpr == 2 ? m >> 1 : m);
                xx = (tpr == 2 ? 128 * (m & 1) : 0) + 32 * quarter + lane;
                valid = yy < H;
            } else {
                const int q = P + 128 * m + 32 * quarter + lane;  // position in brick plane zb = 1
                const int yb = q / P, xp = q - yb * P;
                yy = y0 + yb - 1;
                xx = xp - 1;
                valid = yb >= 1 && yb <= b.Ty && xp >= 1 && xp <= W && yy < H;
            }
            TileVoxel tv;
            tv.valid = valid && ok;
            if (a.y_fp32)
                tv.at = (size_t)t.n * a.nvox + ((size_t)t.z * H + yy) * W + xx;
            else
                tv.at = pg.unit(t.n, Gy, (a.y_coffset + ch) >> 3, t.z, yy, xx);
            if (MODE == kConvMask) tv.mask = pg.unit(t.n, a.mask_cstride >> 3, (a.mask_coffset + ch) >> 3, t.z, yy, xx);
            if (MODE == kConvUp)
                tv.up = Pcg{2 * D, 2 * H, 2 * W}.unit(t.n, a.y_up_cstride >> 3, (a.y_up_coffset + ch) >> 3, 2 * t.z, 2 * yy,
                                                     2 * xx);
            store_columns<MODE>(a, tv, ch, lane, vp, r);
            blk += b.groups;
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    if (tid == 0 && *abort_flag) atomicOr(a.status, 1u);
    if (warp == 0) umma::tmem_dealloc(tbase, (uint32_t)b.tcols);
}

// ----------------------------------------------------------------------------
// Weight gradient: dW[co][tap][ci] = sum over output voxels v of dy[v][co] x[v + off(tap)][ci].
//
// One MMA has K = 16 consecutive positions of an item (Ty rows of one z plane), both operands
// M/N-major core matrices (8 positions x 8 channels), and takes as many of the 27 taps as fit it:
//  - N is the x rows y-1 .. y+1 of the planes z-1 .. z+1 for gpp groups of eight input channels: a
//    plane's slot in shared memory is [gpp][Ty+2][W+2] positions of 16 bytes, exactly the contiguous
//    rows of the padded tensor, and the slots follow each other, so rows, groups and planes all
//    lie at one stride (for Ty = 1 and gpp = 2 nine rows of 16 channels, N = 144);
//  - dx comes from nt offsets t at which the window of x is read, each an accumulator of its own,
//    and from ns copies of the dy row in M, shifted by s positions: dx = s + t.
//
// Two orders of the items (the error of an FP32 sum grows with its K steps, so neither has more of them
// in a sum than the row-block plan):
//  - short sums: a CTA owns a contiguous range of rows (Ty = 1) with z running fastest, so each
//    further row needs one new plane; M is filled with shifted copies (ns = 3 up to 40 channels,
//    2 up to 64), i.e. 96 of its 128 rows at 32 channels;
//  - long sums: the items, K steps and CTAs of the row-block plan in their order, so that every
//    sum is formed from the same products in the same order as with one MMA per tap; three offsets
//    t, no copies.  It keeps those sums, not the better ones: contiguous rows for 32 -> 32 channels on
//    192x128x128 measured 0.30 ms against 0.40 and 2.4e-5 of the largest gradient off the exact one
//    against 4.9e-5, but 3.6e-5 off the row-block plan's sums.
//
// A window of x that passed its row's end would bring other channels' values under the zeros that
// fill dy's last K step, and zero times infinity is no zero.  So the last step's positions lie at its
// end, behind the zeros, and its window starts that much earlier, over positions that are paired
// with zeros there.  A row shorter than a K step has no earlier positions: its passes load one
// group of channels, and the second group's part of each slot stays zero.
//
// Warps 0-7 bring operands, their lanes an item's 10 to 38 bulk copies; warps 8-10 issue the MMAs of
// one offset t each.  They run their loops as whole converged warps, with what one lane alone issues
// predicated: branches for single lanes double the copying warps' time.  A warp issues at some seven
// cycles an instruction, so they keep positions, slots and phases by increments: with the index
// divisions in their loops (three to four thousand cycles an item) they, not the MMAs, set the time.
// An item's commits release its dy slot and the planes no later item needs.  A copying warp waits
// for a slot by the parity of its fillings, so no filling may go by without it: in the long order
// only warps that copy a part of every item take part (without it the item's MMAs cannot run), in
// the short order, where the planes' copies go round the warps, each of them arrives for every
// filling.  dW stays in tensor memory over all of the CTA's items and is added to global memory at
// the end, each CTA starting at another column (all walking the same order would meet on the same
// addresses).
//
// Bound by the MMAs (N / 2 cycles each: the dense rate, a quarter of M used by 32 channels of the
// long sums, three quarters of the short ones).  Before, one MMA a tap with 16 or 32 channels in N
// and the x brick loaded once per tap group: 32 -> 32 channels on 192x128x128 0.915 -> 0.398 ms (long
// order: 0.30 ms of MMAs), 64 -> 96 on 66x54x128 0.316 -> 0.149 ms (short order; 0.117 with the copying
// warps converged).
// ----------------------------------------------------------------------------
constexpr int kRingMaxX = 12, kRingMaxD = 4, kRingCopyWarps = 8, kRingWarps = kRingCopyWarps + 3;

// The MMAs of one item, offset and run of planes, issued by a whole warp's leader.  Unrolled,
// because address arithmetic between two MMAs of one warp costs more than the MMA.
__device__ __forceinline__ void ring_mma(uint32_t leader, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                         uint32_t b_hi, uint32_t idesc, int kst, int back, uint32_t first) {
    umma::mma_bf16_warp(leader, d, a_lo, a_hi, b_lo, b_hi, idesc, first);
    int ks = 1;
    for (; ks + 4 <= kst; ks += 4) {
        const uint32_t last = ks + 4 == kst ? (uint32_t)back : 0u;
#pragma unroll
        for (int u = 1; u <= 4; ++u)
            umma::mma_bf16_warp(leader, d, a_lo + 16 * u, a_hi, b_lo + 16 * u - (u == 4 ? last : 0u), b_hi, idesc, 1u);
        a_lo += 64;
        b_lo += 64;
    }
    for (; ks < kst; ++ks) {
        a_lo += 16;
        b_lo += 16;
        umma::mma_bf16_warp(leader, d, a_lo, a_hi, b_lo - (ks + 1 == kst ? (uint32_t)back : 0u), b_hi, idesc, 1u);
    }
}

// A CTA's items in their order: z plane, row block and sample, by increments.
struct RingItems {
    int left;           // items still to come, this one included
    int z, yb, n;       // z plane, row block, sample
    int sz, syb;        // step in (row block, z plane)
    __device__ __forceinline__ RingItems(const WgradRing& b, int D) {
        const long long G = gridDim.x;
        int item;
        if (b.order) {
            item = blockIdx.x;
            left = (b.items - item + (int)G - 1) / (int)G;
            sz = (int)G % D;
            syb = (int)G / D;
        } else {
            item = (int)(b.items * (long long)blockIdx.x / G);
            left = (int)(b.items * (blockIdx.x + 1ll) / G) - item;
            sz = 1;
            syb = 0;
        }
        z = item % D;
        yb = item / D % b.nyb;
        n = item / D / b.nyb;
    }
    // Whether the next item shares two planes with this one.
    __device__ __forceinline__ bool shares(const WgradRing& b, int D) const { return !b.order && z + 1 < D && left > 1; }
    __device__ __forceinline__ void next(const WgradRing& b, int D) {
        --left;
        z += sz;
        yb += syb;
        if (z >= D) {
            z -= D;
            ++yb;
        }
        for (; yb >= b.nyb; yb -= b.nyb) ++n;
    }
};

// A slot of a ring and the parity of how often the ring was gone round.
struct RingSlot {
    int i = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void advance(int n) {
        if (++i == n) {
            i = 0;
            par ^= 1u;
        }
    }
};

__global__ void __launch_bounds__(32 * kRingWarps, 1) k_wgrad_ring(WgradArgs a, WgradRing b) {
    extern __shared__ __align__(1024) unsigned char smem[];
    // warp-uniform for the compiler too, so that the issuers' operands are
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int Cin = a.Cin, Cout = a.Cout, W = a.W, H = a.H, D = a.D, Yb = b.Ty + 2;
    uint64_t* fullx = reinterpret_cast<uint64_t*>(smem);  // [XS] plane landed
    uint64_t* emptyx = fullx + kRingMaxX;                  // [XS] no later MMA reads the plane
    uint64_t* fulld = emptyx + kRingMaxX;                  // [DS] dy rows landed (long order: planes too)
    uint64_t* emptyd = fulld + kRingMaxD;                  // [DS] item's MMAs finished
    uint64_t* dfull = emptyd + kRingMaxD;                  // all MMAs of the CTA finished
    uint32_t* slot = reinterpret_cast<uint32_t*>(smem + 320);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 324);
    const uint32_t s_d = umma::smem_addr(smem) + kPipeHeader, s_x = umma::smem_addr(smem) + (uint32_t)b.x_off;
    const int c = blockIdx.y;  // chunk of 8 load input channels
    {  // what the copies never write must read as zero, not leftover bits (0 x NaN is NaN)
        uint4* z = reinterpret_cast<uint4*>(smem + kPipeHeader);
        for (int i = tid; i < (b.smem - kPipeHeader) / 16; i += blockDim.x) z[i] = make_uint4(0u, 0u, 0u, 0u);
        umma::fence_async_smem();  // generic-proxy stores -> copies and tensor-core reads
    }
    if (warp == 0) {
        umma::tmem_alloc(slot, 512u);
        umma::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < b.XS; ++i) {
            umma::mbar_init(&fullx[i], (uint32_t)b.arrivals);
            umma::mbar_init(&emptyx[i], b.nt);  // one commit per issuer
        }
        for (int i = 0; i < b.DS; ++i) {
            umma::mbar_init(&fulld[i], (uint32_t)b.arrivals);
            umma::mbar_init(&emptyd[i], b.nt);
        }
        umma::mbar_init(dfull, b.nt);
        *abort_flag = 0;
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tbase = __shfl_sync(0xffffffffu, *slot, 0);
    const int N = 8 * b.ngr;  // columns of an accumulator
    RingItems it(b, D);
    const bool any = it.left > 0;

    if (warp < kRingCopyWarps) {
        // Lanes 0-3 hold the warp's copies of dy rows (copy i = warp + 8 (lane / 2): channel group i % gd of
        // shifted copy i / gd, at most 16 in all; even lanes the whole K steps, odd ones the last
        // step's positions, which go to that step's end), lane 4 in the long order its plane copy (group
        // warp % gpp of plane warp / gpp), and issue them with one instruction.  A lane that waits for a
        // slot has a copy or an arrival in each of its fillings.
        const Pcg pg{D, H, W};
        const int gd = Cout >> 3, nd = b.ns * gd, gx = Cin >> 3;
        const uint32_t xrun = (uint32_t)(Yb * b.P * 16);
        const size_t plane = (size_t)(H + 2) * b.P * 16, vp = pg.vp() * 16;
        const unsigned char* const xsrc =
            reinterpret_cast<const unsigned char*>(a.x + 8 * pg.unit(0, gx, c * b.load, -1, -1, -1));
        const unsigned char* src;  // at z = y0 = n = 0
        uint32_t dst, bytes, slot_step;
        size_t sample;
        bool mine;
        if (lane < 4) {
            const int i = warp + kRingCopyWarps * (lane >> 1), s = i / gd, q = i - s * gd;
            const uint32_t whole = (uint32_t)(b.back ? (b.kst - 1) * 256 : b.drun);
            const bool rest = lane & 1;
            mine = i < nd && (!rest || b.back);
            src = reinterpret_cast<const unsigned char*>(a.dy + 8 * pg.unit(0, gd, q, 0, 0, b.dyx - s)) +
                  (rest ? whole : 0u);
            dst = s_d + (uint32_t)(i * b.ra) + (rest ? whole + 16u * (uint32_t)b.back : 0u);
            bytes = rest ? (uint32_t)b.drun - whole : whole;
            slot_step = (uint32_t)b.dslot;
            sample = (size_t)gd * vp;
        } else {
            const int f = warp / b.gpp, q = warp - f * b.gpp;
            mine = lane == 4 && b.order && f < 3;
            src = xsrc + f * plane + q * vp;
            dst = s_x + (uint32_t)(f * b.xslot) + (uint32_t)q * xrun;
            bytes = xrun;
            slot_step = 3u * (uint32_t)b.xslot;
            sample = (size_t)gx * vp;
        }
        if (warp < b.copiers) {
            RingSlot sd;
            bool ok = true;
            if (b.order) {  // every item brings its three planes, on the dy slot's barrier
                const uint32_t all = (uint32_t)(nd * b.drun) + 3u * (uint32_t)b.gpp * xrun;
                for (int j = 0; it.left > 0; ++j) {
                    if (j >= b.DS) ok = pipe_wait(&emptyd[sd.i], sd.par ^ 1u, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    uint64_t* full = &fulld[sd.i];
                    umma::mbar_arrive_expect_tx_if(tid == 0, full, all);
                    const size_t at = (size_t)it.z * plane + (size_t)(it.yb * b.Ty) * (b.P * 16);
                    umma::bulk_g2s_if(mine, dst + (uint32_t)sd.i * slot_step, src + (at + (size_t)it.n * sample), bytes, full);
                    sd.advance(b.DS);
                    it.next(b, D);
                }
            } else {
                RingSlot sx;
                // fresh: planes this item brings; turn: their copies go round the warps
                int turn = nd, fresh = 3, planes = 0;
                const uint32_t dbytes = warp == 0 ? (uint32_t)(nd * b.drun) : 0u;
                const uint32_t xbytes = warp == 0 ? (uint32_t)b.load * xrun : 0u;
                const unsigned char* const xlane = xsrc + lane * vp;
                const uint32_t xdst = s_x + (uint32_t)lane * xrun;
                for (int j = 0; it.left > 0; ++j) {
                    if (j >= b.DS) ok = pipe_wait(&emptyd[sd.i], sd.par ^ 1u, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    const size_t at = (size_t)it.z * plane + (size_t)it.yb * (b.P * 16);
                    umma::mbar_arrive_expect_tx_if(lane == 0, &fulld[sd.i], dbytes);
                    umma::bulk_g2s_if(mine, dst + (uint32_t)sd.i * slot_step, src + (at + (size_t)it.n * sample), bytes,
                                      &fulld[sd.i]);
                    const unsigned char* xat = xlane + (at + (size_t)it.n * gx * vp + (3 - fresh) * plane);
                    for (int f = 0; f < fresh; ++f, ++planes) {
                        if (planes >= b.XS) ok = pipe_wait(&emptyx[sx.i], sx.par ^ 1u, abort_flag);
                        if (!__all_sync(0xffffffffu, ok)) break;
                        umma::mbar_arrive_expect_tx_if(lane == 0, &fullx[sx.i], xbytes);
                        umma::bulk_g2s_if(lane < b.load && (turn + lane) % kRingCopyWarps == warp,
                                          xdst + (uint32_t)(sx.i * b.xslot), xat, xrun, &fullx[sx.i]);
                        turn += b.load;
                        xat += plane;
                        sx.advance(b.XS);
                    }
                    if (!__all_sync(0xffffffffu, ok)) break;
                    fresh = it.shares(b, D) ? 1 : 3;
                    sd.advance(b.DS);
                    it.next(b, D);
                }
            }
            if (!ok) *abort_flag = 1;  // an expected copy may not come: no one may wait for it
        }
        __syncwarp();
    } else if (warp - kRingCopyWarps < b.nt) {  // issuer of offset t
        const int t = warp - kRingCopyWarps;
        const uint32_t leader = umma::elect_one(), d = tbase + (uint32_t)(t * N);
        // leading byte offset = next 8 positions (K); stride = next 8 channels of dy, next row,
        // 8-channel group or plane of x; descriptors step by their start field, in 16-byte units
        const uint64_t a0 = umma::smem_desc(s_d, 128, (uint32_t)b.ra);
        const uint64_t b0 = umma::smem_desc((uint32_t)((int)s_x + 16 * (b.xoff + t)), 128, (uint32_t)b.P * 16u);
        const uint32_t a_hi = (uint32_t)(a0 >> 32), b_hi = (uint32_t)(b0 >> 32);
        const uint32_t idesc = umma::idesc_bf16_f32(128, N, 1, 1);
        const uint32_t dstep = (uint32_t)b.dslot >> 4, xstep = (uint32_t)b.xslot >> 4;
        RingSlot sd;
        uint32_t accum = 0, a_lo = (uint32_t)a0;
        bool ok = true;
        if (b.order) {
            uint32_t b_lo = (uint32_t)b0;
            for (int left = it.left; left > 0; --left) {
                ok = pipe_wait(&fulld[sd.i], sd.par, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                umma::fence_after_sync();
                ring_mma(leader, d, a_lo, a_hi, b_lo, b_hi, idesc, b.kst, b.back, accum);
                accum = 1;
                umma::mma_commit_warp(leader, &emptyd[sd.i]);
                sd.advance(b.DS);
                a_lo = sd.i ? a_lo + dstep : (uint32_t)a0;
                b_lo = sd.i ? b_lo + 3 * xstep : (uint32_t)b0;
            }
        } else {
            const int gp = b.gpp * Yb;  // row groups of a plane
            RingSlot seen;
            int k = 0, fresh = 3;  // k: slot of the z-1 plane
            while (it.left > 0) {
                for (int f = 0; ok && f < fresh; ++f) {
                    ok = pipe_wait(&fullx[seen.i], seen.par, abort_flag);
                    seen.advance(b.XS);
                }
                ok = ok && pipe_wait(&fulld[sd.i], sd.par, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                umma::fence_after_sync();
                const uint32_t b_lo = (uint32_t)b0 + (uint32_t)k * xstep;
                const int run = b.XS - k;  // planes before the ring wraps
                if (run >= 3) {
                    ring_mma(leader, d, a_lo, a_hi, b_lo, b_hi, idesc, b.kst, b.back, accum);
                } else {
                    const int n1 = run * gp;
                    ring_mma(leader, d, a_lo, a_hi, b_lo, b_hi, umma::idesc_bf16_f32(128, 8 * n1, 1, 1), b.kst, b.back,
                             accum);
                    ring_mma(leader, d + (uint32_t)(8 * n1), a_lo, a_hi, (uint32_t)b0, b_hi,
                             umma::idesc_bf16_f32(128, N - 8 * n1, 1, 1), b.kst, b.back, accum);
                }
                accum = 1;
                umma::mma_commit_warp(leader, &emptyd[sd.i]);
                sd.advance(b.DS);
                a_lo = sd.i ? a_lo + dstep : (uint32_t)a0;
                fresh = it.shares(b, D) ? 1 : 3;
                for (int f = 0; f < fresh; ++f) {
                    umma::mma_commit_warp(leader, &emptyx[k]);
                    k = k + 1 < b.XS ? k + 1 : 0;
                }
                it.next(b, D);
            }
        }
        if (ok) umma::mma_commit_warp(leader, dfull);
        __syncwarp();
    }
    __syncthreads();
    if (*abort_flag) {
        // copies of some item may still be in flight: every barrier's current phase ends when
        // its own copies have landed, or was never armed; wait for the ones that were
        if (tid == 0) {
            for (int i = 0; i < b.DS; ++i)
                for (int ph = 0; ph < 2; ++ph) umma::mbar_wait(&fulld[i], (uint32_t)ph, kWaitCycles >> 6);
            for (int i = 0; i < b.XS; ++i)
                for (int ph = 0; ph < 2; ++ph) umma::mbar_wait(&fullx[i], (uint32_t)ph, kWaitCycles >> 6);
        }
    } else if (warp < 8) {
        bool ok = true;
        if (tid == 0) ok = pipe_wait(dfull, 0u, abort_flag);
        ok = workers_all<256>(ok);
        if (ok && any) {
            umma::fence_after_sync();
            const int quarter = warp & 3;  // tensor-memory lanes 32 quarter .. + 31; two warps share them
            const int m = 32 * quarter + lane, i = m / Cout, co = m - i * Cout;  // row: copy i of channel co
            const bool vec = (reinterpret_cast<uintptr_t>(a.dw) & 15) == 0;
            const int cells = b.nt * b.ngr;  // (offset, row group) cells of eight columns
            if (32 * quarter < b.ns * Cout) {  // warp-uniform: lanes past the last copy load but do not store
                int cell = (int)((blockIdx.x * 7u) % (unsigned)cells);
                for (int n = 0; n < cells; ++n, cell = cell + 1 < cells ? cell + 1 : 0) {
                    if ((n & 1) != (warp >> 2)) continue;
                    const int t = cell / b.ngr, q = cell - t * b.ngr;
                    const int r = q % Yb, pg = q / Yb, dz = pg / b.gpp, g = pg - dz * b.gpp;
                    const int dx = t + i - 1;
                    if (r > 2 || dz > 2 || g >= b.load) continue;  // rows between the taps, groups not loaded
                    float v[8];
                    __syncwarp();
                    umma::tmem_ld8(tbase + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(t * N + 8 * q), v);
                    // two copies give dx = 0 twice, the second time (s = 1, t = -1) without the last position
                    if (i < b.ns && !(b.ns == 2 && i == 1 && t == 0)) {
                        float* d = a.dw + ((size_t)co * 27 + 9 * dz + 3 * r + dx + 1) * Cin + 8 * (c * b.load + g);
                        if (vec) {
                            atomicAdd(reinterpret_cast<float4*>(d), make_float4(v[0], v[1], v[2], v[3]));
                            atomicAdd(reinterpret_cast<float4*>(d) + 1, make_float4(v[4], v[5], v[6], v[7]));
                        } else {
                            for (int e = 0; e < 8; ++e) atomicAdd(d + e, v[e]);
                        }
                    }
                }
            }
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    if (tid == 0 && *abort_flag) atomicOr(a.status, 1u);
    if (warp == 0) umma::tmem_dealloc(tbase, 512u);
}

// wd[ci][26 - tap][co] = w[co][tap][ci]: the data gradient of a 3x3x3 convolution is
// the convolution of dy with these weights.
__global__ void k_flip_weights(const __nv_bfloat16* w, __nv_bfloat16* wd, int Cin, int Cout) {
    const int n = Cout * 27 * Cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int ci = i % Cin, tap = (i / Cin) % 27, co = i / (27 * Cin);
        wd[((size_t)ci * 27 + (26 - tap)) * Cout + co] = w[i];
    }
}

}  // namespace

// Work decomposition of the pipelined brick kernel for one layer shape: output channels
// split into parts of Cp, weights resident or streamed, rows per item Ty (the last row block
// may pass H), and for 128-voxel rows the x-tap fold, by a cost model.  Its constants are per-role
// cycle counts of an earlier kernel, which had two epilogue groups of whole tiles and one-thread
// roles; they have not been measured again for the present one, nor does the model know waves, so
// its choices are only as good as these: a tcgen05.mma (M = 128, K = 16) took ~64 cycles of one
// issuing thread at N = 32, ~85 at N = 64, ~90 at N = 96 and about N / 2 from N = 192, less with two
// issuers (mma_pair_factor); bulk copies of brick runs moved ~64 bytes per cycle per SM; the
// epilogue took ~700 cycles per tile and 8 columns (~850 folded) on each of two warp groups and
// overlapped the MMAs only with two accumulators; copies and MMAs overlapped, but not perfectly
// (a quarter of the shorter one showed).
static double mma_cycles(int N) {
    return N <= 32 ? 64.0 : (N <= 64 ? 85.0 : (N <= 96 ? 90.0 : (N <= 192 ? 96.0 + (N - 128) / 2.0 : N / 2.0)));
}
// Time per MMA with two issuers relative to one (microbenchmark: 65 cycles from one thread,
// (4 KB of A + N x 32 bytes of B) / 128 bytes per cycle from two, at least the dense peak).
static double mma_pair_factor(int N) {
    const double two = (4096.0 + 32.0 * N) / 128.0, peak = 2.0 * 128 * N * 16 / 8192.0;
    return (two > peak ? two : peak) / 65.0 < 1.0 ? (two > peak ? two : peak) / 65.0 : 1.0;
}

static bool brick_plan(int D, int H, int W, int Cin, int Cout, int batch, BrickPlan* out, size_t* smem_out) {
    const int P = W + 2;
    const size_t smem_cap = 227 * 1024;
    const bool rowtile = W % 128 == 0;
    double best = 1e300;
    bool found = false;
    const int nchunk = Cin / 16;
    for (int nsplit = 1; nsplit <= Cout / 16; ++nsplit) {
        if (Cout % nsplit || (Cout / nsplit) % 16) continue;
        const int Cp = Cout / nsplit;
        if (Cp > 256) continue;
        const size_t w_bytes = (size_t)27 * Cp * 32;
        for (int fold = 0; fold <= (W == 128 && 3 * Cp <= 256 ? 1 : 0); ++fold)
            for (int wres = nsplit == 1 ? 1 : 0; wres >= 0; --wres)  // ties keep the weights resident
                for (int Ty = 1; Ty <= H; ++Ty) {
                    const int nyb = (H + Ty - 1) / Ty;
                    const int tiles = rowtile ? Ty * (W / 128) : (Ty * P + 127) / 128;
                    const int cols = tiles * Cp * (fold ? 3 : 1);  // accumulator columns per item
                    if (cols > 512 || tiles > (fold ? 4 : 8)) break;  // the MMA loops are unrolled up to these
                    const int nacc = 2 * cols <= 512 ? 2 : 1;
                    const size_t run = (size_t)(Ty + 2) * P * 16;
                    const size_t plane = (3 * run + 127) / 128 * 128;
                    // flat tiles read up to 128 positions past the end of the second plane
                    const size_t w_off = (128 + 2 * plane + (rowtile ? 0 : 2048) + 127) / 128 * 128;
                    const size_t stage = wres ? w_off : (w_off + w_bytes + 127) / 128 * 128;
                    const size_t xch = kPipeHeader + kPipeStages * stage + (wres ? nchunk * w_bytes : 0);
                    const size_t smem = xch + (fold ? (size_t)128 * Cp : 0);
                    if (smem > smem_cap || plane >= (1u << 18)) break;
                    // two issuers share the tiles: pairs of tiles at the two-issuer rate, an odd
                    // last tile at one issuer's
                    const int Nmma = fold ? 3 * Cp : Cp;
                    const double per_tile = (fold ? 9 : 27) * mma_cycles(Nmma);
                    const double mma = (double)nchunk * per_tile * ((tiles / 2) * 2 * mma_pair_factor(Nmma) + tiles % 2);
                    const double load = (double)nchunk * (6 * run + (wres ? 0 : w_bytes)) / 64.0;
                    const double epi = ((tiles + 1) / 2) * (Cp / 8.0) * (fold ? 850.0 : 700.0);
                    double item = (mma > load ? mma : load) + 0.25 * (mma > load ? load : mma);
                    item = nacc == 2 ? (item > epi ? item : epi) : item + epi;
                    const double cost = item * nyb / ((double)H * W) * nsplit;  // per output voxel, all parts
                    if (cost < best) {
                        best = cost;
                        found = true;
                        int tcols = 32;
                        while (tcols < nacc * cols) tcols <<= 1;
                        BrickPlan bp{};
                        bp.Ty = Ty;
                        bp.tiles = tiles;
                        bp.rowtile = rowtile ? 1 : 0;
                        bp.fold = fold;
                        bp.nyb = nyb;
                        bp.P = P;
                        bp.Yb = Ty + 2;
                        bp.Cp = Cp;
                        bp.nsplit = nsplit;
                        bp.plane = (int)plane;
                        bp.w_off = (int)w_off;
                        bp.wres = wres;
                        bp.stage = (int)stage;
                        bp.nacc = nacc;
                        bp.xch = (int)xch;
                        bp.tcols = tcols;
                        bp.items = batch * nsplit * nyb * D;
                        const int turns = nacc * tiles * (Cp / 16);
                        bp.groups = turns < kConvGroups ? turns : kConvGroups;
                        *out = bp;
                        *smem_out = smem;
                    }
                }
    }
    return found;
}

// Element of wpk = [part][chunk][tap][core-matrix image of the Cp x 16 tile] that holds
// w[co][tap][ci] of a layer of Cin input channels.
__device__ __forceinline__ size_t packed_at(int co, int tap, int ci, int Cin, int Cp) {
    const int part = co / Cp, r = co - part * Cp;
    const size_t tile = (((size_t)part * (Cin >> 4) + (ci >> 4)) * 27 + tap) * Cp * 16;
    return tile + umma::core_offset(r, ci & 15, 16) / 2;
}

static __global__ void k_pack_weights(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wpk, int Cin,
                               int Cout, int Cp) {
    const int n = Cout * 27 * Cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int ci = i % Cin, tap = (i / Cin) % 27, co = i / (27 * Cin);
        wpk[packed_at(co, tap, ci, Cin, Cp)] = w[i];
    }
}

static __global__ void k_pack_network(const __grid_constant__ PackNet net) {
    const int l = blockIdx.y, Cin = net.Cin[l], Cout = net.Cout[l], n = Cout * 27 * Cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int ci = i % Cin, tap = (i / Cin) % 27, co = i / (27 * Cin);
        const __nv_bfloat16 v = net.w[l][i];
        net.fwd[l][packed_at(co, tap, ci, Cin, net.cp[l])] = v;
        if (net.bwd[l]) net.bwd[l][packed_at(ci, 26 - tap, co, Cout, net.cpf[l])] = v;
    }
}

cudaError_t conv_pack_network(const PackNet& net, int layers, cudaStream_t st) {
    k_pack_network<<<dim3(128, (unsigned)layers), 256, 0, st>>>(net);
    return cudaGetLastError();
}

int conv_plan_cp(int D, int H, int W, int Cin, int Cout) {
    BrickPlan bp{};
    size_t smem = 0;
    return brick_plan(D, H, W, Cin, Cout, 1, &bp, &smem) ? bp.Cp : 0;
}

cudaError_t conv_pack_weights(const __nv_bfloat16* w, __nv_bfloat16* wpk, int Cin, int Cout, int Cp,
                              cudaStream_t st) {
    if (Cp <= 0 || Cout % Cp || Cin % 16) return cudaErrorInvalidValue;
    k_pack_weights<<<256, 256, 0, st>>>(w, wpk, Cin, Cout, Cp);
    return cudaGetLastError();
}

cudaError_t conv3d_launch(const ConvArgs& a, int batch, cudaStream_t st) {
    BrickPlan bp{};
    size_t bsmem = 0;
    if (!brick_plan(a.D, a.H, a.W, a.Cin, a.Cout, batch, &bp, &bsmem) || bp.Cp != a.wpk_cp)
        return cudaErrorInvalidValue;
    auto* kernel = a.y_up   ? k_conv3d_brick<kConvUp>
                   : a.mask ? k_conv3d_brick<kConvMask>
                            : k_conv3d_brick<kConvPlain>;
    if (a.y_up && a.mask) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsmem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int ctas = bp.items < sms ? bp.items : sms;
    kernel<<<ctas, kConvThreads, bsmem, st>>>(a, bp);
    return cudaGetLastError();
}

// Row-block plan of the weight gradient (sde_conv3d_wgrad_plan): Nc in {16, 32} input channels
// per pass, as many taps per pass as 512 tensor-memory columns hold, and Ty a divisor of H whose
// two stages fit.  It was the launched decomposition before the rings below; the shapes that the
// call accepts are still those that it has a plan for.
static bool wgrad_plan(const WgradArgs& a, int sms, WgradPlan* out, size_t* smem_out) {
    const int P = a.W + 2;
    double best = 1e300;
    bool found = false;
    for (int Nc = 16; Nc <= 32; Nc += 16) {
        if (a.Cin % Nc) continue;
        const int ntap = Nc == 16 ? 27 : 14;
        const int ngroups = (27 + ntap - 1) / ntap;
        for (int Ty = 1; Ty <= a.H; ++Ty) {
            if (a.H % Ty) continue;
            const int kst = (Ty * P + 15) / 16;
            const size_t plane_dy = (size_t)kst * 256;
            const size_t dy_bytes = (size_t)(a.Cout / 8) * plane_dy;
            const size_t plane_x = ((size_t)3 * (Ty + 2) * P * 16 + 127) / 128 * 128;
            const size_t x_off = (dy_bytes + 16 + 127) / 128 * 128;  // >= 16 bytes before the brick
            size_t stage = (x_off + (size_t)(Nc / 8) * plane_x + 512 + 127) / 128 * 128;
            if (stage < 16 * plane_dy) stage = (16 * plane_dy + 127) / 128 * 128;  // A rows past Cout stay inside
            const size_t smem = kPipeHeader + kPipeStages * stage;
            if (smem > 227 * 1024 || plane_x >= (1u << 18) || plane_dy >= (1u << 18)) break;
            const double pos = (double)Ty * a.W;  // output voxels per item
            const double mma = (double)kst * 27 * 56.0 * (a.Cin / Nc);
            const double bytes = (double)(a.Cout / 8) * Ty * P * 16 + (double)(Nc / 8) * 3 * (Ty + 2) * P * 16;
            const double load = bytes / 64.0 * (a.Cin / Nc) * ngroups;
            const double cost = (mma > load ? mma : load) / pos;
            if (cost < best) {
                best = cost;
                found = true;
                const int nyb = a.H / Ty;
                const int items = a.batch * nyb * a.D;
                const int passes = (a.Cin / Nc) * ngroups;
                // CTAs per pass: all passes in one wave on the SMs (a CTA past it would run its
                // whole share again after the others)
                int G = sms / passes > 1 ? sms / passes : 1;
                if (G > items) G = items;
                *out = WgradPlan{Ty, nyb, P, Ty + 2, Nc, ntap, ngroups, kst, (int)plane_dy, (int)plane_x,
                                 (int)x_off, (int)stage, items, G};
                *smem_out = smem;
            }
        }
    }
    return found;
}

// Rings of the weight gradient for one layer shape: the order of the items by the length of its
// sums (in K steps of the row-block plan), then as many dy slots (up to four) and plane slots (up
// to twelve; the fewer, the more often a range's planes wrap) as fit.  At 1024 steps the short
// order's gradient differs from the row-block plan's by about 1.2e-5 of its largest value, without
// being less exact, and takes half the time of the long one.
constexpr double kLongSum = 1024.0;

bool wgrad_ring_plan(const WgradArgs& a, int sms, const WgradPlan& wp, WgradRing* out) {
    const double steps = (double)wp.items / wp.G * wp.kst;
    for (int order = steps > kLongSum && wp.Ty <= 6 ? 1 : 0; order >= 0; --order) {
        WgradRing w{};
        w.order = order;
        w.P = a.W + 2;
        if (order) {
            w.Ty = wp.Ty;
            w.ns = 1;
            // what three accumulators in tensor memory leave room for; one where a K step passes the rows
            w.gpp = wp.Ty == 1 && wp.kst > 1 ? 2 : 1;
            w.kst = wp.kst;
            w.drun = w.Ty * w.P * 16;  // rows with their padding, from x = -1
            w.dyx = -1;
            w.G = wp.G;
        } else {
            w.Ty = 1;
            w.ns = a.Cout <= 40 ? 3 : a.Cout <= 64 ? 2 : 1;
            // always two groups of channels: where the ring wraps inside a window the MMA is cut into runs
            // of gpp Yb row groups, and with one group these would be 24 and 56 columns, which an
            // MMA of M = 128 does not take (multiples of 16)
            w.gpp = 2;
            w.kst = (a.W + 15) / 16;
            w.drun = a.W * 16;
            w.dyx = w.ns == 3 ? 1 : 0;  // copy 0 is shifted by s = -1 or 0
        }
        const int used = w.drun / 16 - 16 * (w.kst - 1);  // positions of the last K step
        w.back = w.kst > 1 ? 16 - used : 0;
        w.load = w.kst > 1 || used == 16 ? w.gpp : 1;
        w.nt = w.ns == 3 ? 1 : w.ns == 2 ? 2 : 3;
        // the window of t = t0 at the first position: the slot's rows start at x = -1
        w.xoff = order ? -1 : w.nt == 1 ? 1 : 0;
        w.nyb = a.H / w.Ty;
        w.items = a.batch * w.nyb * a.D;
        const int Yb = w.Ty + 2, passes = a.Cin / (8 * w.load);
        w.ngr = ((3 * w.gpp - 1) * Yb + 3 + 1) / 2 * 2;  // N is a multiple of 16
        w.ra = w.kst * 256;
        w.dslot = w.ns * (a.Cout / 8) * w.ra;
        w.xslot = w.gpp * Yb * w.P * 16;
        if (!order) {
            // all passes in one wave on the SMs, or in as many as it takes for sums no longer than the
            // row-block plan's: the error of an FP32 sum grows with its K steps, and narrow rows, whose
            // K steps hold one row each, have up to five times as many of them (192 -> 32 on
            // 192x128x24: 7.5e-5 of the largest gradient off in one wave, 3.9e-5 in two; 1.28 and 1.51 ms, 1.05
            // in two with the copying warps converged)
            const int one = sms / passes > 1 ? sms / passes : 1;
            const long long most = (long long)((wp.items + wp.G - 1) / wp.G) * wp.kst;
            for (w.G = std::min(one, w.items); w.G < w.items; w.G = std::min(w.G + one, w.items))
                if ((long long)((w.items + w.G - 1) / w.G) * w.kst <= most) break;
        }
        for (w.DS = kRingMaxD; w.DS >= 2; --w.DS)
            for (w.XS = order ? 3 * w.DS : kRingMaxX; w.XS >= (order ? 3 * w.DS : w.DS + 2); --w.XS) {
                w.x_off = kPipeHeader + w.DS * w.dslot;
                // the windows of the last three slots may end past them (with rows of 256 and 64 or 128
                // output channels a more generous end leaves no room for four planes), and M = 128 rows
                // of A start in the last dy slot
                const int past = (w.ngr - 1) * w.P + w.xoff + w.nt - 1 + 16 * w.kst - 3 * w.xslot / 16;
                const int tail = kPipeHeader + (w.DS - 1) * w.dslot + 16 * w.ra;
                w.smem = w.x_off + w.XS * w.xslot + (past > 0 ? past : 0) * 16;
                if (w.smem < tail) w.smem = tail;
                if (w.smem <= 227 * 1024) {
                    const int nd = w.ns * (a.Cout / 8);
                    w.copiers = order ? std::min(kRingCopyWarps, std::max(nd, 3 * w.gpp)) : kRingCopyWarps;
                    w.arrivals = order ? 1 : w.copiers;
                    *out = w;
                    return true;
                }
            }
    }
    return false;
}

cudaError_t wgrad_launch(const WgradArgs& a, cudaStream_t st) {
    WgradPlan wp{};
    WgradRing wr{};
    size_t wsmem = 0;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (!wgrad_plan(a, sms, &wp, &wsmem) || !wgrad_ring_plan(a, sms, wp, &wr)) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(k_wgrad_ring, cudaFuncAttributeMaxDynamicSharedMemorySize, wr.smem);
    if (e != cudaSuccess) return e;
    k_wgrad_ring<<<dim3((unsigned)wr.G, (unsigned)(a.Cin / (8 * wr.load))), 32 * kRingWarps, wr.smem, st>>>(a, wr);
    return cudaGetLastError();
}

}  // namespace sde

static bool conv_shape_ok(int D, int H, int W, int Cin, int Cout, int batch) {
    const long long vp = (long long)(D + 2) * (H + 2) * (W + 2);
    return batch >= 1 && D >= 1 && H >= 1 && W >= 1 && W <= 256 && vp * batch * 256 < (1ll << 40) && Cin >= 16 &&
           Cin <= 192 && Cin % 16 == 0 && Cout >= 16 && Cout <= 256 && Cout % 16 == 0;
}

extern "C" int sde_conv3d_forward(const void* d_x, int batch, int D, int H, int W, int Cin, const void* d_w,
                                  const float* d_bias, int Cout, void* d_y, int y_cstride, int y_coffset,
                                  int y_fp32, int relu, void* stream) {
    if (!d_x || !d_w || !d_y || !conv_shape_ok(D, H, W, Cin, Cout, batch) || y_cstride < Cout + y_coffset ||
        y_coffset < 0 || (y_coffset % 8) || (y_cstride % 8) ||
        (((uintptr_t)d_x | (uintptr_t)d_y | (uintptr_t)d_bias) & 15)) {
        set_last_error("sde_conv3d_forward: need W <= 256, Cin in 16..192 and Cout in 16..256 (multiples of 16), "
                       "y_cstride >= Cout + y_coffset, both multiples of 8, 16-byte aligned x, y and bias");
        return SDE_EINVAL;
    }
    unsigned int* d_status = nullptr;
    int rc = report(status_word(&d_status), "status word");
    if (rc) return rc;
    const int Cp = conv_plan_cp(D, H, W, Cin, Cout);
    if (!Cp) {
        set_last_error("sde_conv3d_forward: no tile plan fits shared memory for this shape");
        return SDE_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    __nv_bfloat16* wpk = nullptr;  // weights in the tensor core's layout, stream-ordered scratch
    rc = report(scratch_alloc(reinterpret_cast<void**>(&wpk), (size_t)Cout * 27 * Cin * 2, st), "scratch allocation");
    if (rc) return rc;
    rc = report(conv_pack_weights(static_cast<const __nv_bfloat16*>(d_w), wpk, Cin, Cout, Cp, st), "pack weights");
    ConvArgs a;
    a.x = static_cast<const __nv_bfloat16*>(d_x);
    a.wpk = wpk;
    a.wpk_cp = Cp;
    a.bias = d_bias;
    a.y = d_y;
    a.D = D;
    a.H = H;
    a.W = W;
    a.Cin = Cin;
    a.Cout = Cout;
    a.nvox = D * H * W;
    a.y_cstride = y_cstride;
    a.y_coffset = y_coffset;
    a.y_fp32 = y_fp32;
    a.y_keep = 0;
    a.y_up = nullptr;
    a.y_up_cstride = a.y_up_coffset = 0;
    a.mask = nullptr;
    a.mask_cstride = a.mask_coffset = 0;
    a.mask_slope = 0.f;
    a.relu = relu;
    a.slope = 0.f;
    a.status = d_status;
    if (!rc) rc = report(conv3d_launch(a, batch, st), "conv3d launch");
    const int rf = report(cudaFreeAsync(wpk, st), "cudaFreeAsync");
    return rc ? rc : rf;
}

extern "C" int sde_conv3d_wgrad(const void* d_x, const void* d_dy, float* d_dw, int batch, int D, int H, int W,
                                int Cin, int Cout, void* stream) {
    if (!d_x || !d_dy || !d_dw || !conv_shape_ok(D, H, W, Cin, Cout, batch) || Cout > 128 ||
        (((uintptr_t)d_x | (uintptr_t)d_dy) & 15)) {
        set_last_error("sde_conv3d_wgrad: need W <= 256, Cin in 16..192, Cout in 16..128 (multiples of 16), "
                       "16-byte aligned x and dy");
        return SDE_EINVAL;
    }
    unsigned int* d_status = nullptr;
    int rc = report(status_word(&d_status), "status word");
    if (rc) return rc;
    WgradArgs a;
    a.x = static_cast<const __nv_bfloat16*>(d_x);
    a.dy = static_cast<const __nv_bfloat16*>(d_dy);
    a.dw = d_dw;
    a.D = D;
    a.H = H;
    a.W = W;
    a.Cin = Cin;
    a.Cout = Cout;
    a.nvox = D * H * W;
    a.batch = batch;
    a.status = d_status;
    return report(wgrad_launch(a, (cudaStream_t)stream), "wgrad launch");
}

extern "C" int sde_conv3d_flip_weights(const void* d_w, void* d_wd, int Cin, int Cout, void* stream) {
    if (!d_w || !d_wd || Cin < 1 || Cout < 1) {
        set_last_error("sde_conv3d_flip_weights: bad arguments");
        return SDE_EINVAL;
    }
    k_flip_weights<<<256, 256, 0, (cudaStream_t)stream>>>(static_cast<const __nv_bfloat16*>(d_w),
                                                            static_cast<__nv_bfloat16*>(d_wd), Cin, Cout);
    return report(cudaGetLastError(), "k_flip_weights launch");
}

extern "C" int sde_denoise_status(void* stream) { return denoise_check_status((cudaStream_t)stream); }

// Host-only views of the two plans (no CUDA call).
extern "C" int sde_conv3d_plan(int batch, int D, int H, int W, int Cin, int Cout, int32_t* fields, int n_fields,
                               uint64_t* smem_bytes) {
    BrickPlan bp{};
    size_t smem = 0;
    if (!conv_shape_ok(D, H, W, Cin, Cout, batch) || n_fields < 0 || (n_fields > 0 && !fields) ||
        !brick_plan(D, H, W, Cin, Cout, batch, &bp, &smem)) {
        set_last_error("sde_conv3d_plan: shape rejected by the convolution or without a plan");
        return SDE_EINVAL;
    }
    const int32_t v[18] = {bp.Ty,    bp.tiles, bp.rowtile, bp.fold,  bp.nyb, bp.P,    bp.Yb,  bp.Cp,   bp.nsplit,
                           bp.plane, bp.w_off, bp.wres,    bp.stage, bp.nacc, bp.xch, bp.tcols, bp.items, bp.groups};
    for (int i = 0; i < n_fields && i < 18; ++i) fields[i] = v[i];
    if (smem_bytes) *smem_bytes = smem;
    return SDE_OK;
}

extern "C" int sde_conv3d_wgrad_plan(int batch, int D, int H, int W, int Cin, int Cout, int sms, int32_t* fields,
                                     int n_fields, uint64_t* smem_bytes) {
    WgradArgs a{};
    a.D = D;
    a.H = H;
    a.W = W;
    a.Cin = Cin;
    a.Cout = Cout;
    a.nvox = D * H * W;
    a.batch = batch;
    WgradPlan wp{};
    size_t smem = 0;
    if (!conv_shape_ok(D, H, W, Cin, Cout, batch) || Cout > 128 || sms < 1 || n_fields < 0 ||
        (n_fields > 0 && !fields) || !wgrad_plan(a, sms, &wp, &smem)) {
        set_last_error("sde_conv3d_wgrad_plan: shape rejected by the weight gradient or without a plan");
        return SDE_EINVAL;
    }
    const int32_t v[14] = {wp.Ty,       wp.nyb,     wp.P,     wp.Yb,    wp.Nc,    wp.ntap,  wp.ngroups,
                           wp.kst,      wp.plane_dy, wp.plane_x, wp.x_off, wp.stage, wp.items, wp.G};
    for (int i = 0; i < n_fields && i < 14; ++i) fields[i] = v[i];
    if (smem_bytes) *smem_bytes = smem;
    return SDE_OK;
}

extern "C" int sde_conv3d_wgrad_ring(int batch, int D, int H, int W, int Cin, int Cout, int sms, int32_t* fields,
                                     int n_fields, uint64_t* smem_bytes) {
    WgradArgs a{};
    a.D = D;
    a.H = H;
    a.W = W;
    a.Cin = Cin;
    a.Cout = Cout;
    a.nvox = D * H * W;
    a.batch = batch;
    WgradRing w{};
    WgradPlan wp{};
    size_t smem = 0;
    if (!conv_shape_ok(D, H, W, Cin, Cout, batch) || Cout > 128 || sms < 1 || n_fields < 0 ||
        (n_fields > 0 && !fields) || !wgrad_plan(a, sms, &wp, &smem) || !wgrad_ring_plan(a, sms, wp, &w)) {
        set_last_error("sde_conv3d_wgrad_ring: shape rejected by the weight gradient or without a plan");
        return SDE_EINVAL;
    }
    const int32_t v[23] = {w.order, w.Ty,    w.gpp,   w.ngr, w.ns, w.nt,    w.kst,   w.P, w.ra,      w.drun,    w.dyx,
                           w.xoff,  w.dslot, w.xslot, w.DS,  w.XS, w.x_off, w.items, w.G, w.copiers, w.arrivals,
                           w.load,  w.back};
    for (int i = 0; i < n_fields && i < 23; ++i) fields[i] = v[i];
    if (smem_bytes) *smem_bytes = (uint64_t)w.smem;
    return SDE_OK;
}
