// Host-side shared declarations of the library: context, status helpers, kernel launchers.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <unordered_map>
#include <vector>

#include "../../include/b2c.h"

// Bits of the sticky device status word.
#define B2C_DEV_TIMEOUT 1u
#define B2C_DEV_BAD_LABEL 2u

typedef CUresult (*b2c_encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                        const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                        CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// What a launch plan depends on, as words that compare and hash in a few instructions (the look-up is on the path of every launch).
struct b2c_plan_key {
    unsigned long long w[16];
    bool operator==(const b2c_plan_key& o) const
    {
        unsigned long long d = 0;
        for (int i = 0; i < 16; ++i) d |= w[i] ^ o.w[i];
        return d == 0;
    }
};
struct b2c_plan_key_hash {
    size_t operator()(const b2c_plan_key& k) const
    {
        unsigned long long h = 0x9e3779b97f4a7c15ull;
        for (int i = 0; i < 16; ++i) h = (h ^ k.w[i]) * 0x100000001b3ull + (h >> 29);
        return (size_t)(h ^ (h >> 32));
    }
};
static inline unsigned long long b2c_key_pair(int a, int b) { return ((unsigned long long)(unsigned)a << 32) | (unsigned)b; }
static inline unsigned long long b2c_key_ptr(const void* p) { return (unsigned long long)reinterpret_cast<uintptr_t>(p); }

struct b2c_ctx {
    int device;
    int sm_count;
    unsigned* d_status;  // one device word
    unsigned spin_limit;
    b2c_encode_tiled_fn encode_tiled;
    int use_full_halo;                   // 3x3 stride-1 convolutions with a resident filter bank stage one framed tile for all nine taps
    int use_pairs;                       // forward / data-gradient convolutions may run on CTA pairs (cta_group::2)
    unsigned long long* stall_counters;  // optional device array the convolution kernels add their wait cycles to
    int use_wgrad_frame;                 // weight gradient of 3x3 stride-1 layers stages x once per chunk with a one-pixel frame (all three shifts from one box)
    int use_issue_split;                 // forward / data-gradient tiles wider than 128 channels: two MMA-issuing threads share every unit
    int use_pdl;                         // kernels are launched with programmatic stream serialization (their set-up overlaps the previous kernel's tail)
    int use_hmerge;                      // forward / data gradient of 3x3 stride-1 layers with 64 output channels: horizontal taps merged into N = 192 MMAs
    int use_group_kblocks;               // short k-blocks of stride-2 and 1x1 layers share ring slots (fewer barrier waits per MMA)
    int use_split_k;                     // forward / data gradient with up to two tiles per SM: one wave, clusters of CTAs may share a tile's k-blocks (conv_splitk.cu)
    int max_clusters[2][9];              // clusters of 1..8 CTAs that run at once, for single CTAs and pairs; -1: not asked yet
    int use_wgrad_two_issuers;           // weight gradient: two MMA-issuing threads on alternate chunks of one accumulator where the ring depth is even
    int use_bn_grouped;                  // BatchNorm backward of the training step: both passes in one cooperative launch, group by group
    // Launch plans (kernel parameter blocks with their tensor maps, grid and shared-memory size) of the convolution
    // kernels, keyed by the problem description: pointers and shapes of a bound network repeat every
    // step, so a plan is built once and its launches cost one parameter copy.
    std::unordered_map<b2c_plan_key, std::vector<unsigned char>, b2c_plan_key_hash> plan_cache;
    unsigned smem_optin_done;            // kernels whose dynamic shared-memory opt-in was set on this context's device (B2C_OPTIN_* bits)
};
#define B2C_OPTIN_KMAJOR 1u
#define B2C_OPTIN_WGRAD 2u
#define B2C_OPTIN_BN_BWD 4u
#define B2C_OPTIN_BN_GROUPED 8u
#define B2C_OPTIN_SPLITK 16u

#define B2C_CUDA(call)                               \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return B2C_ERR_CUDA;  \
    } while (0)

// Kernel launch.  With ctx->use_pdl the launch carries the programmatic-stream-serialization attribute: the kernel may be
// scheduled while the previous kernel of the stream drains, and it orders itself behind that kernel with pdl_wait() before its first
// global access; convolutions launched with no_wait do so at their end (pdl_begin, pdl_end).  cluster > 1 launches thread-block clusters.
template <typename... KArgs, typename... Args>
static inline cudaError_t b2c_launch(const b2c_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     unsigned cluster, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (ctx->use_pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

static inline bool b2c_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline bool b2c_is_pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }

namespace b2c {

// Filter taps of one launch: which tensor map (parity view) a tap gathers from, its pixel
// offset inside that view, and its index in the weight tensor's tap dimension.
struct TapList {
    int count;
    int8_t map[9], dh[9], dw[9], rs[9];
};

// bf16 activation tensor [n][h][w][c] as a 4-D tensor map (c, w/step, h/step, n); step 2 selects
// rows of parity ph and columns of parity pw.  Box = (box_c, box_w, box_h, box_n); swizzle = box_c*2 bytes.
bool encode_activation_map(b2c_ctx* ctx, CUtensorMap* tm, const void* base, int n, int h, int w, int c, int step, int ph, int pw, int box_c,
                           int box_w, int box_h, int box_n);
// Taps of a forward convolution in terms of (parity view, offset): input row = p*stride + r - pad.
void forward_taps(TapList& tl, int R, int stride, int pad);

// Geometry of one implicit-GEMM launch with K-major operands (forward and data gradient):
// the "input" is the activation tensor that is gathered (x for fprop, dy for dgrad), the
// "output" the tensor that is written.  in_pitch / out_pitch are channel strides in elements.
struct KMajorProblem {
    int n;                 // images
    int ih, iw, ic;        // gathered tensor
    int oh, ow, oc;        // written tensor
    int r, stride, pad;    // filter taps (r x r), forward stride and padding of the convolution
    bool dgrad;            // false: forward; true: data gradient (input = dy, weights in [c,r,s,k] flipped layout)
    const void* in;
    const void* wt;        // [oc][r*r][ic] bf16
    void* out;
    bool out_f32;
    const float* bias;
    double* stats;         // fp64 [groups][2*oc] or nullptr
    int stats_group_images;  // images per statistics group (0: one group)
    // Data gradient whose output is the last contribution to the gradient of a BatchNorm(+ReLU) output: `stats` takes the sums of the BatchNorm's
    // backward pass, sum dz and sum dz*y with dz = (out + bwd_other) where bwd_mask has a bit, else 0.  A plan that cannot ignores them.
    const void* bwd_y;       // the BatchNorm's input (nullptr: no such sums)
    const void* bwd_other;   // the other contribution, or nullptr
    const void* bwd_mask;    // one bit per element, or nullptr
    bool* bwd_done;          // set to whether the launch takes the sums
    bool ask_sums;         // a question about the plan of a call with `stats`
    bool no_wait;          // the launch right before this one shares nothing that is written with this one, and itself waits for the one before it
                           // (it is not no_wait): the kernel starts as SMs fall free and waits for that launch only at its end
};
b2c_status launch_conv_kmajor(b2c_ctx* ctx, const KMajorProblem& pb, cudaStream_t stream);
// Whether a forward convolution with BatchNorm sums works in blocks in its epilogue.  Asks the planner, without launching anything; for problems
// of more than two units per CTA it asks the device nothing.
bool kmajor_sums_in_blocks(b2c_ctx* ctx, KMajorProblem pb);
b2c_status plan_conv_kmajor(b2c_ctx* ctx, const KMajorProblem& pb, b2c_conv_plan_detail& out);   // pointers of the problem: null

struct WgradProblem {
    int n, h, w, c;        // x
    int p, q, k;           // dy
    int r, stride, pad;
    const void* dy;
    const void* x;
    float* dw;             // [k][r*r][c] fp32, accumulated into
};
b2c_status launch_conv_wgrad(b2c_ctx* ctx, const WgradProblem& pb, cudaStream_t stream);
b2c_status plan_conv_wgrad(b2c_ctx* ctx, const WgradProblem& pb, b2c_conv_plan_detail& out);

// BatchNorm over G statistics groups (micro-batches) of m rows each; stats / sums are fp64 [G][2c],
// save_mean / save_invstd fp32 [G][c].  G > 1 requires acc != 0 in the backward pass.  stats_ready: 1 = `stats` holds the
// sums already (convolution epilogue), 0 = clear and compute them, 2 = compute them into `stats` the caller has cleared.  relu_mask (optional): one bit per
// element, "stored output > 0" (a byte per 8 channels), written by the forward pass and read by the backward pass
// in place of the output tensor.  sums_ready: `sums` holds the sums already (a data gradient's epilogue).  sums_zeroed: the caller has already cleared `sums` (and `arrivals`).  arrivals (optional): G
// zeroed counters; with them the two passes run in one cooperative launch, group by group (bn_bwd_grouped_kernel).
b2c_status launch_bn_fwd(b2c_ctx* ctx, int G, long long m, int c, const void* y, double* stats, int stats_ready, const float* gamma,
                         const float* beta, const void* residual, int relu, float eps, void* a, float* save_mean, float* save_invstd,
                         float* run_mean, float* run_var, float momentum, void* relu_mask, cudaStream_t stream);
b2c_status launch_bn_bwd(b2c_ctx* ctx, int G, long long m, int c, const void* da1, const void* da2, const void* y, const void* a,
                         const float* gamma, const float* save_mean, const float* save_invstd, int relu, void* dy, void* dres, float* dgamma,
                         float* dbeta, int acc, double* sums, bool sums_ready, bool sums_zeroed, const void* relu_mask, unsigned* arrivals, cudaStream_t stream);

// Average + SGD-momentum update of `count` elements, gradient sums cleared, and both bf16 copies, in one launch.  The segments (filter banks)
// lie back to back from element 0 and their sizes are multiples of 8; elements behind the last one have no data-gradient layout.
b2c_status launch_update_pack(b2c_ctx* ctx, const b2c_weight_seg* segs, int n_segs, size_t count, float* w, float* v, float* g, float inv_n, float lr, float momentum,
                              float wd, void* w_bf16, void* w_dgrad, cudaStream_t stream);

// Clears `bytes` (a multiple of 8, 8-byte aligned) at `a` and, if f is not null, one float, as a launch like any other of the stream.
b2c_status launch_zero(b2c_ctx* ctx, void* a, size_t bytes, float* f, cudaStream_t stream);

// Running statistics of the BatchNorm layers of a step (momentum update with the unbiased variance), taken from the fp64
// sums the forward pass left in the workspace.  One entry per layer; the G statistics groups of a pass are applied in
// order, as if the micro-batches had run one after the other.
struct BnRunEntry {
    long long stats_off;   // bytes into the workspace: fp64 [G][2c] sum / sum of squares
    int c;                 // channels
    int run_off;           // elements into the running-statistics array: [mean c][var c]
    float m;               // rows per group
};
b2c_status launch_bn_running_update(b2c_ctx* ctx, const BnRunEntry* entries, int n_entries, const char* ws, float* run, int G, float momentum,
                                    cudaStream_t stream);

}  // namespace b2c
