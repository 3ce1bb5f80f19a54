// Parameter block and unit numbering shared by the two implicit-GEMM kernels with K-major operands: the persistent one
// (conv_kmajor.cu) and the split-K one for problems with up to one or two tiles per SM (conv_splitk.cu).  The packed arithmetic
// serves both, the column exchanges behind it the persistent one.
#pragma once
#include "common.h"
#include "ptx.cuh"

namespace b2c {

struct alignas(64) ConvKParams {
    CUtensorMap tmA[4];
    CUtensorMap tmB;
    TapList taps[4];
    int bw, bh, bn;                  // pixel box of an output tile; bw*bh*bn == 128
    int tiles_w, tiles_h, tiles_n;   // tiles of the output grid
    int tw_shift, th_shift, nk_shift, grp_shift, cb_shift;   // log2 of tiles_w, tiles_h, n_ktiles, stats_group_images, c_blocks (-1: not a power of two)
    int n_ktiles, n_tile;            // output-channel tiles, UMMA N
    int n_par;                       // output parities (stride-2 data gradient: 4)
    int total_units;
    int kb, c_blocks;                // channels per k-block, k-blocks per tap
    int stages, swz;
    int tmem_cols, acc_cols;         // allocation, columns per accumulator
    int acc_bufs, acc_shift;         // accumulators in TMEM (2 or 4) and log2 of that: unit j uses accumulator j % acc_bufs
    int vreuse;                      // a stage serves the three vertical taps of one horizontal shift
    int fh;                          // full halo: a stage holds the tile with a one-pixel frame and serves all nine taps
    int hm;                          // merged horizontal taps: one N = 3 x n_tile MMA per vertical tap and k-step, the three column blocks are
                                     // shifted by one pixel and added in the epilogue (tiles of whole image rows, 64 output channels)
    int mma_n;                       // UMMA N (n_tile, or 3 x n_tile with merged horizontal taps)
    int nb;                          // B tiles per stage (1, or 3 with vreuse)
    int b_merged;                    // the three B tiles of a stage come with one load (box of three filter rows)
    int r_filter;                    // filter height = width
    int a_bytes, b_bytes;            // shared-memory footprint of the A tile / one B tile (multiples of 1 KB)
    int tx_a, tx_b;                  // bytes one A / B load delivers
    int a_step;                      // byte offset of one image row inside the A tile (vreuse)
    int issuers;                     // MMA-issuing threads at work (1 or 2)
    int gsub;                        // k-blocks that share a ring slot, one barrier wait and one commit (short k-blocks: the waits would bound the issuing threads)
    int issue_split;                 // the two issuing threads share every unit: alternate stages into one accumulator (tiles wider than 128 channels)
    int splits;                      // split-K plans (conv_splitk.cu): CTAs (or CTA pairs) of a cluster that share a unit's k-blocks; 0: persistent kernel
    int x_off, x_overlap;            // split-K: byte offset of the exchange area behind the ring's start; it overlaps the ring
    int pair;                        // CTA pairs (cta_group::2): M = 256 per MMA, each CTA holds half of every B tile
    int block_cols;                  // columns that an epilogue warp turns from a row per lane into rows of 16-byte vectors at a time (0: it does not)
    int resident;                    // filter bank of this CTA's channel tile stays in shared memory
    int resident_bytes;
    int n_valid, oc_valid;           // images / output channels that exist
    long long os_n, os_h, os_w;      // output element strides along the tile grid
    int row_bit[7];                  // output elements between rows m and m + 2^i of a tile (its sides are powers of two: bits of m add up)
    long long off[4];                // output element offset per parity
    void* out;
    int out_is_f32;
    int out_v8;                      // the output base is 32-byte aligned: bf16 chunks go out as one 256-bit store per lane
    const float* bias;
    double* stats;
    int stats_group_images;          // images per BatchNorm statistics group (0: one group)
    const void *bwd_y, *bwd_other;   // sums of a BatchNorm's backward pass in place of those of the output (see KMajorProblem)
    const uint8_t* bwd_mask;
    int no_wait;                     // starts beside the previous launch of the stream, see pdl_begin
    unsigned* status;
    unsigned spin_limit;
    unsigned long long* stall;       // optional [5]: cycles waited by producer / MMA (ring) / MMA (accumulator) / epilogue, CTA lifetime
};

struct UnitCoord {
    int par, ktile, ow0, oh0, n0;
};
// tiles_w and tiles_h are powers of two (the grid sides are); the channel-tile count and the stats group size usually are
__device__ __forceinline__ UnitCoord decode_unit(const ConvKParams& p, int u)
{
    UnitCoord c;
    if (p.nk_shift >= 0) {
        c.ktile = u & (p.n_ktiles - 1);
        u >>= p.nk_shift;
    } else {
        c.ktile = u % p.n_ktiles;
        u /= p.n_ktiles;
    }
    c.ow0 = (u & (p.tiles_w - 1)) * p.bw;
    u >>= p.tw_shift;
    c.oh0 = (u & (p.tiles_h - 1)) * p.bh;
    u >>= p.th_shift;
    if (p.n_par > 1) {
        c.n0 = (u % p.tiles_n) * p.bn;
        c.par = u / p.tiles_n;
    } else {
        c.n0 = u * p.bn;
        c.par = 0;
    }
    return c;
}

// Two fp32 values in a register pair and the packed arithmetic on them (one issue slot for two adds or fused multiply-adds).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 make_f32x2(float lo, float hi)
{
    f32x2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 split_f32x2(f32x2 v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ f32x2 add_f32x2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul_f32x2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma_f32x2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 widen_bf16x2(uint32_t pair) { return make_f32x2(__uint_as_float(pair << 16), __uint_as_float(pair & 0xffff0000u)); }
// s += both values of a packed bf16 pair, q += their squares.
__device__ __forceinline__ void add_pair(uint32_t pair, f32x2& s, f32x2& q)
{
    const f32x2 f = widen_bf16x2(pair);
    s = add_f32x2(s, f);
    q = fma_f32x2(f, f, q);
}

// Adds a warp's 32 rows x 16 columns of stored bf16 values (packed pairs pk, one row per lane, rows that do not exist as zeros) to
// the lane's sums s and sums of squares q.  Two exchanges of packed pairs leave a lane with four columns of four rows, so a chunk needs
// four register pairs for its sums instead of sixteen: lane l holds columns 8 (l >> 4) + 4 (l >> 3 & 1) + {0, 1} in s[0], q[0] and
// + {2, 3} in s[1], q[1], and the eight lanes that differ in the lower bits are added up by column_total.
__device__ __forceinline__ void add_chunk(const uint32_t (&pk)[8], int lane, f32x2 (&s)[2], f32x2 (&q)[2])
{
    const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
    uint32_t half[2][4];   // [row: own, the partner's][pair]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        half[0][i] = up16 ? pk[4 + i] : pk[i];
        half[1][i] = __shfl_xor_sync(0xffffffffu, up16 ? pk[i] : pk[4 + i], 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        f32x2 f[4];   // four rows of the lane's column pair
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            f[2 * r] = widen_bf16x2(up8 ? half[r][2 + i] : half[r][i]);
            f[2 * r + 1] = widen_bf16x2(__shfl_xor_sync(0xffffffffu, up8 ? half[r][i] : half[r][2 + i], 8));
        }
        s[i] = add_f32x2(s[i], add_f32x2(add_f32x2(f[0], f[1]), add_f32x2(f[2], f[3])));
        q[i] = add_f32x2(q[i], add_f32x2(fma_f32x2(f[1], f[1], mul_f32x2(f[0], f[0])), fma_f32x2(f[3], f[3], mul_f32x2(f[2], f[2]))));
    }
}
__device__ __forceinline__ float2 column_total(f32x2 v)
{
    float2 f = split_f32x2(v);
#pragma unroll
    for (int bit = 1; bit <= 4; bit <<= 1) {
        f.x += __shfl_xor_sync(0xffffffffu, f.x, bit);
        f.y += __shfl_xor_sync(0xffffffffu, f.y, bit);
    }
    return f;
}
__device__ __forceinline__ int column_of(int lane) { return (lane & 24) >> 1; }   // first of a lane's four columns; lanes with (l & 7) == 0 speak for them

// Column sums over the 32 rows a warp holds (one row per lane, 16 columns each): a butterfly that halves the
// number of columns each lane carries (16 -> 8 -> 4 -> 2 -> 1).  On return lane l holds in a[0], b[0] the totals of
// column (l >> 1) of the chunk.
__device__ __forceinline__ void butterfly16(float (&a)[16], float (&b)[16], int lane)
{
#pragma unroll
    for (int width = 8, bit = 16; width >= 1; width >>= 1, bit >>= 1) {
        const bool upper = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < width; ++i) {
            const float sa = upper ? a[i] : a[i + width], ka = upper ? a[i + width] : a[i];
            const float sb = upper ? b[i] : b[i + width], kb_ = upper ? b[i + width] : b[i];
            a[i] = ka + __shfl_xor_sync(0xffffffffu, sa, bit);
            b[i] = kb_ + __shfl_xor_sync(0xffffffffu, sb, bit);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    b[0] += __shfl_xor_sync(0xffffffffu, b[0], 1);
}

// What the sums of a BatchNorm's backward pass need of 8 neighbouring elements.  The loads pass the L1 by: a launch that starts beside the one
// before it (no_wait) may find lines there that are older than its operands.
struct BwdVec {
    uint4 y, other;
    unsigned mask;
};
__device__ __forceinline__ void bwd_load(const ConvKParams& p, long long element, BwdVec& v)
{
    v.y = __ldcg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.bwd_y) + element));
    v.other = p.bwd_other != nullptr ? __ldcg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.bwd_other) + element)) : make_uint4(0u, 0u, 0u, 0u);
    v.mask = p.bwd_mask != nullptr ? (unsigned)__ldcg(p.bwd_mask + (element >> 3)) : 0xffu;
}
// dz of columns 2 k and 2 k + 1 of such a vector, from the packed pair that the convolution stores there.
__device__ __forceinline__ f32x2 bwd_pair(uint32_t stored, uint32_t other, unsigned mask, int k)
{
    const float2 f = split_f32x2(add_f32x2(widen_bf16x2(stored), widen_bf16x2(other)));
    return make_f32x2((mask >> (2 * k)) & 1u ? f.x : 0.f, (mask >> (2 * k + 1)) & 1u ? f.y : 0.f);
}
__device__ __forceinline__ uint32_t word_of(const uint4& v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// Clusters of `cluster` CTAs (pair: made of CTA pairs) that run at the same time on this context's device.
int splitk_max_clusters(b2c_ctx* ctx, int cluster, bool pair);
// Split-K plan: the parameter block, CTAs per cluster and in all, dynamic shared memory.
b2c_status launch_conv_splitk(b2c_ctx* ctx, const ConvKParams& p, int grid, size_t smem_bytes, cudaStream_t stream);

}  // namespace b2c
