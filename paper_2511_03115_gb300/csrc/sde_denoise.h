// sde_denoise.h -- internal interface of the denoiser's tensor-core kernels.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace sde {

// Activation layout of the denoiser ("padded channel-group-major"): a BF16 tensor of C
// channels on a D x H x W grid is stored as [n][C/8][D+2][H+2][W+2][8], i.e. per group of
// eight channels a zero-padded volume whose voxels hold 16 bytes.  The one-voxel border is
// the convolutions' zero padding: it is zeroed when the buffer is created and no kernel
// writes it.  In this layout the rows y0-1 .. y0+Ty of one padded plane of one channel
// group are a single contiguous run of (Ty+2)(W+2) x 16 bytes, which one bulk copy moves
// into exactly the shared-memory image the tensor core reads.
struct Pcg {
    int D, H, W;
    __host__ __device__ size_t vp() const { return (size_t)(D + 2) * (H + 2) * (W + 2); }
    // 16-byte unit of voxel (z, y, x) (interior coordinates, -1 .. D etc. reach the border)
    // of channel group g of sample n, in a tensor of G groups
    __host__ __device__ size_t unit(int n, int G, int g, int z, int y, int x) const {
        return ((((size_t)n * G + g) * (D + 2) + (z + 1)) * (H + 2) + (y + 1)) * (W + 2) + (x + 1);
    }
};

// 3x3x3 convolution as an implicit GEMM (see sde_denoise.cu).  x is padded
// channel-group-major with Cin channels; the BF16 output is padded channel-group-major
// with y_cstride channels (written from channel y_coffset on), the FP32 output plain
// channels-last [n][D H W][y_cstride].  wpk holds the weights packed for the tensor core
// with wpk_cp output channels per part (conv_pack_weights; the plan's Cp must match).
struct ConvArgs {
    const __nv_bfloat16* x;
    const __nv_bfloat16* wpk;
    int wpk_cp;
    const float* bias;
    void* y;
    int D, H, W, Cin, Cout;
    int nvox;  // D*H*W
    int y_cstride, y_coffset, y_fp32, relu;
    int y_keep;   // FP32 output only: > 0 stores just output channels 0 .. y_keep-1 (<= 16), dense [n][D H W][y_keep]
    // BF16 output only, optional: also store every output voxel to its eight children in a padded
    // channel-group-major tensor on the grid 2D x 2H x 2W (nearest-neighbour upsampling), at
    // channel y_up_coffset of y_up_cstride
    void* y_up;
    int y_up_cstride, y_up_coffset;
    // BF16 output only, optional: the adjoint of a leaky ReLU on the stored values, which are multiplied
    // by mask_slope where mask (channels mask_coffset .. of mask_cstride, the activation's output) is
    // not positive
    const __nv_bfloat16* mask;
    int mask_cstride, mask_coffset;
    float mask_slope;
    float slope;  // with relu: y = x > 0 ? x : slope * x (0: ReLU, > 0: leaky ReLU)
    unsigned int* status;
};

// Work decomposition and shared-memory layout of the pipelined brick convolution
// (host-chosen per layer shape).  A work item is (sample, Cout part, row block, z plane).
struct BrickPlan {
    int Ty;       // output rows (y) per work item, all x of one z plane (the last block may pass H)
    int tiles;    // M tiles of 128 positions per work item
    int rowtile;  // 1: W is a multiple of 128 and each tile is 128 x of one output row
    int fold;     // 1 (row tiles only): the three x taps of a (z, y) tap pair in one MMA of N = 3 Cp
    int nyb;      // ceil(H / Ty)
    int P;        // W + 2: brick row pitch in positions
    int Yb;       // Ty + 2: brick rows per plane
    int Cp;       // output channels per work item
    int nsplit;   // Cout / Cp
    int plane;    // bytes between the two 8-channel planes of a 16-channel chunk
    int w_off;    // offset of the chunk's weights (27 taps x Cp x 16) within a stage (wres = 0)
    int wres;     // 1: all chunks' weights stay resident after the stages (loaded once per CTA)
    int stage;    // bytes per pipeline stage (brick chunk + weight chunk)
    int nacc;     // tensor-memory accumulators (2: epilogue overlaps the next item)
    int xch;      // fold: offset of the epilogue's boundary-exchange buffer in shared memory
    int tcols;    // tensor-memory columns allocated (power of two >= nacc x tiles x Cp x (fold ? 3 : 1))
    int items;    // batch x nsplit x nyb x D
    int groups;   // epilogue groups that take part: at most nacc x tiles x Cp/16
};

// Weight gradient of the convolution; x and dy padded channel-group-major.
struct WgradArgs {
    const __nv_bfloat16* x;   // Cin channels
    const __nv_bfloat16* dy;  // Cout channels
    float* dw;                // [Cout][27][Cin], accumulated
    int D, H, W, Cin, Cout, nvox, batch;
    unsigned int* status;
};

// Work decomposition of the brick weight-gradient kernel (host-chosen).  A pass is one
// chunk of Nc input channels and one group of taps (its accumulators fill tensor memory);
// a work item is Ty output rows of one z plane.
struct WgradPlan {
    int Ty, nyb, P, Yb;  // as BrickPlan
    int Nc;              // input channels per pass (MMA N)
    int ntap, ngroups;   // taps per pass, tap groups
    int kst;             // K steps (16 positions) per item
    int plane_dy;        // bytes between 8-channel planes of the output-gradient rows
    int plane_x;         // bytes between 8-channel planes of the input brick
    int x_off;           // offset of the input brick within a stage
    int stage;           // bytes per stage
    int items;           // batch x nyb x D
    int G;               // CTAs per pass
};

// Order, rings and operand shapes of the weight-gradient kernel (host-chosen per layer shape).
struct WgradRing {
    int order;         // 0: contiguous rows per CTA (short sums), 1: the row-block plan's items (long sums)
    int Ty, nyb;       // rows per item, H / Ty
    int gpp;           // groups of eight input channels in a plane slot
    int ngr;           // row groups of N (N = 8 ngr)
    int ns;            // copies of the dy row in M, shifted by s = -1..1 (3), 0..1 (2) or 0 (1)
    int nt;            // offsets at which the x window is read: 0 (1), -1..0 (2) or -1..1 (3)
    int kst;           // K steps of 16 positions per item
    int P;             // W + 2: positions of an x row
    int ra;            // bytes of an 8-channel run of dy (kst x 16 positions)
    int drun, dyx;     // bytes copied into it, x of its first position in copy 0
    int xoff;          // position in a plane's first row under the item's first position, at the first offset
    int dslot, xslot;  // bytes of a dy slot (ns x Cout/8 runs) and of a plane slot (gpp x (Ty + 2) rows)
    int DS, XS;        // dy slots and plane slots
    int x_off;         // offset of the first plane slot
    int smem;          // dynamic shared memory in bytes
    int items;         // batch x nyb x D
    int G;             // CTAs per pass
    int copiers;       // copying warps that take part
    int load;          // channel groups loaded per pass: gpp, or 1 (the others stay zero)
    int back;          // positions by which the last K step's window starts before the step: it ends with the dy row
    int arrivals;      // arrivals per filling of a slot: 1 (every copier has a part of each), or all copiers
};

// Output channels per part that conv3d_launch will use for this layer shape (the packing
// of its weights), or 0 if the shape has no plan.
int conv_plan_cp(int D, int H, int W, int Cin, int Cout);
// wpk = w [Cout][27][Cin] in the tensor core's shared-memory image:
// [Cout/Cp][Cin/16][27][Cp x 16 K-major core matrices].
cudaError_t conv_pack_weights(const __nv_bfloat16* w, __nv_bfloat16* wpk, int Cin, int Cout, int Cp, cudaStream_t st);
// The packed images of a whole network's layers in one launch: fwd[i] = w[i] as conv_pack_weights
// packs it with cp[i] channels per part, and where bwd[i] is not NULL the weights of the data
// gradient (wd[ci][26 - tap][co] = w[co][tap][ci]) with cpf[i].
struct PackNet {
    static constexpr int kMaxLayers = 16;
    const __nv_bfloat16* w[kMaxLayers];
    __nv_bfloat16* fwd[kMaxLayers];
    __nv_bfloat16* bwd[kMaxLayers];
    int Cin[kMaxLayers], Cout[kMaxLayers], cp[kMaxLayers], cpf[kMaxLayers];
};
cudaError_t conv_pack_network(const PackNet& net, int layers, cudaStream_t st);
cudaError_t conv3d_launch(const ConvArgs& a, int batch, cudaStream_t st);
cudaError_t wgrad_launch(const WgradArgs& a, cudaStream_t st);
cudaError_t denoise_status_word(unsigned int** out);
int denoise_check_status(cudaStream_t st);
// Gives the scratch pool's unused memory on the current device back.
void denoise_scratch_trim();

}  // namespace sde
