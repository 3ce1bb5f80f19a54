// Implicit-GEMM convolution for problems with up to one output tile per SM (two, where they are small): forward pass, data
// gradient and classifier at small batches.
//
// The operands, tap tables and tile geometry are those of conv_kmajor.cu; what differs is the split of the work.  There, a
// CTA owns a whole tile, so a layer with 16 tiles of 72 k-blocks runs 72 k-blocks in a row on 16 SMs (or pairs) and leaves
// the rest idle: 512 -> 512 channels at 4x4 with 128 images took 28 us, of which 19.4 us were the 36.8 k cycles of one
// pair's MMAs.  Here a cluster of `splits` CTAs (or CTA pairs) shares a tile: each accumulates its share of the k-blocks in
// its own TMEM, then the partial tiles are added up through distributed shared memory, every CTA finishing one slice of the
// columns.  Nothing is written to global memory but the result, so no workspace and no second launch are needed.
//   * One tile per cluster, not persistent: barriers and TMEM are set up once, every warp joins the epilogue when the main
//     loop has been issued, and the kernel is small (a launch inside a step starts on a cold instruction cache).
//   * The exchange has an area of its own where three or four ring slots fit beside it; otherwise it goes through the ring's
//     memory, which is free once the MMAs of every CTA of the cluster have completed (one more cluster barrier, about 1350
//     cycles).  A lane holds one row, so a block of four columns is stored as 128 rows x 16 bytes: neighbouring lanes write
//     neighbouring 16-byte words of the receiver, and the next columns are read from TMEM while the current ones are sent.
//   * A slot holds two or four k-blocks of a narrow tile: waiting, issuing and committing cost about 500 cycles per slot, as
//     long as the MMAs of 256 channels (128 channels, 36 k-blocks: 19.8 k cycles to the last MMA with one k-block per slot,
//     13.4 k with two).
// What bounds it now: the operands' way from L2 (about 74 B/clk per SM), then the set-up and the exchange, about 3 us together.
// Launch to launch with 128 images: 512 -> 512 at 4x4 28 us in the persistent kernel, 13.6 here (17.4 with one k-block per slot,
// the exchange in the ring and single-buffered); 256 -> 256 at 8x8 18.2 and 12.3 (14.1); the ResNet-18-shaped step of 128 images
// 1.89 -> 1.73 ms when this kernel came and 1.490 -> 1.452 ms with those three, as four micro-batches of 50 6.32 -> 5.41 and
// 4.41 -> 4.28 ms.
// Warp roles during the main loop: warp 0 = TMA producer, warp 1 = TMEM owner and MMA issuer.  Every mbarrier wait is
// bounded; a CTA that gives up still takes part in both cluster barriers.
#include "conv_kmajor.h"

namespace b2c {

static constexpr int kSkThreads = 256;
static constexpr int kSkStages = 8;
static constexpr uint32_t kSkDrainPolls = 1u << 22;

template <bool PAIR>
__device__ __forceinline__ void sk_issue(int ksteps, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc, uint32_t accumulate_first)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k >= ksteps) break;
        const uint64_t ad = ((uint64_t)desc_hi << 32) | (uint64_t)(a_lo + 2u * k), bd = ((uint64_t)desc_hi << 32) | (uint64_t)(b_lo + 2u * k);
        if constexpr (PAIR) umma_bf16_pair(d_tmem, ad, bd, idesc, k == 0 ? accumulate_first : 1u);
        else umma_bf16(d_tmem, ad, bd, idesc, k == 0 ? accumulate_first : 1u);
    }
}

// BatchNorm sums of a warp's 32 rows x 16 columns of stored bf16 values (packed pairs, one row per lane, rows that do not exist as
// zeros).  The block goes through 1 KB of shared memory as [half][row][8 columns]; ldmatrix with transposition then hands lane l eight
// rows of column l >> 2 of each half, which it adds up in fp32, and the four lanes of a column share the rest: on return the lane holds
// one total, of column column_of_total(l): the sum, or the sum of squares if total_is_square(l).
// The squares of bf16 values end in the same few bits, so a running sum loses a quarter of a unit in its last place with every other
// addition, always downwards; here four squares meet exactly or nearly so before anything larger is added.  On the tensor cores, whose
// accumulators truncate, the sums of squares came out 5.0e-8 low; now 1.1e-8 off, as in the persistent kernel.
__device__ __forceinline__ int column_of_total(int lane) { return 8 * (lane & 1) + (lane >> 2); }
__device__ __forceinline__ int total_is_square(int lane) { return (lane >> 1) & 1; }
__device__ __forceinline__ float column_sums(const uint32_t (&pk)[8], float* stage, int lane)
{
    const uint32_t base = smem_u32(stage) + 16u * (uint32_t)lane;
    __syncwarp();   // the previous block has been read
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]) : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + 512u), "r"(pk[4]), "r"(pk[5]), "r"(pk[6]), "r"(pk[7]) : "memory");
    __syncwarp();
    float s[2], q[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t t[4];   // t[i]: rows 8 i + 2 (lane & 3) + {0, 1} of column lane >> 2
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3])
                     : "r"(base + 512u * h)
                     : "memory");
        const f32x2 f0 = widen_bf16x2(t[0]), f1 = widen_bf16x2(t[1]), f2 = widen_bf16x2(t[2]), f3 = widen_bf16x2(t[3]);
        const float2 ss = split_f32x2(add_f32x2(add_f32x2(f0, f1), add_f32x2(f2, f3)));
        const float2 qq = split_f32x2(add_f32x2(fma_f32x2(f1, f1, mul_f32x2(f0, f0)), fma_f32x2(f3, f3, mul_f32x2(f2, f2))));
        s[h] = ss.x + ss.y;
        q[h] = qq.x + qq.y;
    }
    // four totals over four lanes: each exchange halves what a lane carries
    const bool odd = (lane & 1) != 0, upper = (lane & 2) != 0;
    const float ms = (odd ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, odd ? s[0] : s[1], 1);
    const float mq = (odd ? q[1] : q[0]) + __shfl_xor_sync(0xffffffffu, odd ? q[0] : q[1], 1);
    return (upper ? mq : ms) + __shfl_xor_sync(0xffffffffu, upper ? ms : mq, 2);
}

// TIMED: the instance that adds to the stall counters (read at run time, they cost the small net of tests and benchmarks 2.5 % of
// its step: 198 -> 203 us)
// BWD: the instance that takes the sums of a BatchNorm's backward pass (p.bwd_y), with shuffles: its products are fp32.  A launch of 6-8 us that
// reads the gradient again is replaced by 2-4 us in this one (the first operands come in while the accumulator is waited for).  Steps: two
// blocks of 64 and 128 channels on 16x16, 16 images, 162.4 -> 148.5 us, ResNet-18-shaped 128 images 1327 -> 1309, 4 x 50 images 3786 -> 3679.
template <bool PAIR, bool TIMED, bool BWD>
__global__ void __launch_bounds__(kSkThreads, 1) conv_splitk_kernel(const __grid_constant__ ConvKParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kSkStages], empty_bar[kSkStages], acc_bar, drain_bar;
    __shared__ uint32_t tmem_slot, abort_flag;
    __shared__ float s_sum[4][2][256];   // BatchNorm sums of this CTA's columns, per TMEM lane quarter (shared-memory float atomics took 500 cycles a block)
    __shared__ __align__(16) float s_stage[kSkThreads / 32][256];   // staging of column_sums

    // (the same offset in every CTA of the cluster: the exchange maps addresses from one CTA to another)
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~uintptr_t(1023));
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int cta = p.splits * (PAIR ? 2 : 1) > 1 ? (int)cluster_ctarank() : 0;
    const int rank = PAIR ? cta & 1 : 0;                // CTA of its pair: 0 issues the MMAs and owns the pair's barriers
    const int split = PAIR ? cta >> 1 : cta;
    const uint32_t leader = (uint32_t)(cta - rank);
    const int S = p.stages, G = p.gsub;
    const int sub_bytes = p.a_bytes + p.b_bytes, stage_bytes = G * sub_bytes;

    const long long t_start = TIMED ? clock64() : 0;

    // the unit of this cluster (a pair takes two neighbouring pixel tiles) and this CTA's share of its k-blocks
    const int cluster_id = (int)blockIdx.x / (p.splits * (PAIR ? 2 : 1));
    const UnitCoord c = decode_unit(p, PAIR ? (2 * (cluster_id / p.n_ktiles) + rank) * p.n_ktiles + cluster_id % p.n_ktiles : cluster_id);
    const TapList& tl = p.taps[c.par];
    const int k_total = tl.count * p.c_blocks;
    const int k_begin = k_total * split / p.splits, k_count = k_total * (split + 1) / p.splits - k_begin;
    const int n_slots = (k_count + G - 1) / G;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&acc_bar, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            tmem_alloc_pair(&tmem_slot, (uint32_t)p.tmem_cols);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(&tmem_slot, (uint32_t)p.tmem_cols);
            tmem_relinquish();
        }
    } else if (warp == 0 && elect_one()) {
        prefetch_tensormap(&p.tmB);
        prefetch_tensormap(&p.tmA[tl.map[0]]);
    }
    tc_fence_before();
    __syncthreads();
    const bool clustered = PAIR || p.splits > 1;
    if (clustered) cluster_sync_all();   // the others' barriers and memory exist before anything arrives there
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    pdl_begin(p.no_wait);

    int issued = 0;   // producer warp: ring slots whose loads it has issued
    if (warp == 0) {
        const int R = p.r_filter, b_rows = PAIR ? p.n_tile >> 1 : p.n_tile;
        const int oc0 = c.ktile * p.n_tile + rank * b_rows;
        int s = 0;
        uint32_t ph = 0;
        long long waited = 0;
        for (int it = 0; it < n_slots; ++it) {
            const long long t0 = TIMED ? clock64() : 0;
            if (!mbar_wait_warp(&empty_bar[s], ph ^ 1u, p.spin_limit, &abort_flag)) {
                if (lane == 0) atomicOr(p.status, B2C_DEV_TIMEOUT);
                break;
            }
            if (TIMED) waited += clock64() - t0;
            const int n_k = k_count - it * G < G ? k_count - it * G : G;
            if (elect_one()) {
                const uint32_t bar = PAIR ? map_to_cta(smem_u32(&full_bar[s]), leader) : 0u;
                if (rank == 0) mbar_expect_tx(&full_bar[s], (PAIR ? 2u : 1u) * (uint32_t)(n_k * (p.tx_a + p.tx_b)));   // a pair counts both CTAs' bytes
                for (int g = 0; g < n_k; ++g) {
                    const int kblk = k_begin + it * G + g;
                    const int tap = p.cb_shift >= 0 ? kblk >> p.cb_shift : kblk / p.c_blocks, cb = kblk - tap * p.c_blocks;
                    const int rs = tl.rs[tap], fr = (rs * 11) >> 5;   // rs / 3 for rs < 9 (R is 1 or 3)
                    uint8_t* dst = ring + (size_t)s * stage_bytes + (size_t)g * sub_bytes;
                    if constexpr (PAIR) {
                        tma_load_4d_pair(dst, &p.tmA[tl.map[tap]], bar, cb * p.kb, c.ow0 + tl.dw[tap], c.oh0 + tl.dh[tap], c.n0);
                        tma_load_4d_pair(dst + p.a_bytes, &p.tmB, bar, cb * p.kb, rs - fr * R, oc0, fr);
                    } else {
                        tma_load_4d(dst, &p.tmA[tl.map[tap]], &full_bar[s], cb * p.kb, c.ow0 + tl.dw[tap], c.oh0 + tl.dh[tap], c.n0);
                        tma_load_4d(dst + p.a_bytes, &p.tmB, &full_bar[s], cb * p.kb, rs - fr * R, oc0, fr);
                    }
                }
            }
            __syncwarp();
            issued = it + 1;
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (TIMED && rank == 0 && lane == 0) atomicAdd(p.stall + 0, (unsigned long long)waited);
    } else if (warp == 1 && rank == 0) {
        const uint32_t idesc = make_idesc_bf16(PAIR ? 256 : 128, p.n_tile, false, false);
        const uint64_t proto = make_smem_desc(0u, 16u, 8u * (uint32_t)p.kb * 2u, (uint32_t)p.swz);   // eight rows of kb bf16
        const uint32_t desc_hi = (uint32_t)(proto >> 32), ring_lo = (uint32_t)proto + (smem_u32(ring) >> 4);
        const uint32_t a_to_b16 = (uint32_t)p.a_bytes >> 4, sub16 = (uint32_t)sub_bytes >> 4, stage16 = (uint32_t)stage_bytes >> 4;
        const int ksteps = p.kb >> 4;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        long long waited = 0;
        for (int it = 0; it < n_slots; ++it) {
            const long long t0 = TIMED ? clock64() : 0;
            ok = mbar_wait_warp(&full_bar[s], ph, p.spin_limit, &abort_flag);
            if (!ok) {
                if (lane == 0) atomicOr(p.status, B2C_DEV_TIMEOUT);
                break;
            }
            if (TIMED) waited += clock64() - t0;
            tc_fence_after();
            const int n_k = k_count - it * G < G ? k_count - it * G : G;
            if (elect_one()) {
                uint32_t a_lo = ring_lo + (uint32_t)s * stage16;
                for (int g = 0; g < n_k; ++g, a_lo += sub16)
                    sk_issue<PAIR>(ksteps, tmem_base, a_lo, a_lo + a_to_b16, desc_hi, idesc, (it | g) != 0 ? 1u : 0u);
                if constexpr (PAIR) umma_commit_pair(&empty_bar[s], (uint16_t)(3u << leader));
                else umma_commit(&empty_bar[s]);
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (TIMED && lane == 0) atomicAdd(p.stall + 1, (unsigned long long)waited);
        if (ok && n_slots > 0 && elect_one()) {
            if constexpr (PAIR) umma_commit_pair(&acc_bar, (uint16_t)(3u << leader));
            else umma_commit(&acc_bar);
        }
        __syncwarp();
    }

    // ---------------------------------------------------------------- epilogue: all eight warps
    const int q = warp & 3, half = warp >> 2;   // TMEM lane quarter of this warp, half of the columns
    const int m = q * 32 + lane;                // accumulator row = pixel of the tile (w fastest, then h, then image)
    const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
    const int sw = p.n_tile / p.splits;         // columns this CTA finishes
    const int col0 = split * sw;
    const int lw = m % p.bw, lh = (m / p.bw) % p.bh, ln = m / (p.bw * p.bh);
    const bool row_valid = c.n0 + ln < p.n_valid;
    const long long row_off = (long long)(c.n0 + ln) * p.os_n + (long long)(c.oh0 + lh) * p.os_h + (long long)(c.ow0 + lw) * p.os_w + p.off[c.par];
    // 16 columns at a time (the last step of an odd count of eights takes 8)
    const int n16 = (sw + 15) >> 4, g_lo = half ? (n16 + 1) >> 1 : 0, g_hi = half ? n16 : (n16 + 1) >> 1;
    // what the sums of a BatchNorm's backward pass need beside the output: read a step ahead, the first step's before the accumulator is waited for
    BwdVec in[2];
    auto load_bwd = [&](int g) {
        const long long at = row_off + c.ktile * p.n_tile + col0 + g * 16;
        in[0] = in[1] = BwdVec{make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u), 0u};
        if (row_valid) {
            bwd_load(p, at, in[0]);
            if (g * 16 + 16 <= sw) bwd_load(p, at + 8, in[1]);
        }
    };
    if (BWD && g_lo < g_hi) load_bwd(g_lo);
    const long long t_wait = TIMED ? clock64() : 0;
    if (n_slots > 0 && !mbar_wait_warp(&acc_bar, 0u, p.spin_limit, &abort_flag) && lane == 0) atomicOr(p.status, B2C_DEV_TIMEOUT);
    if (TIMED && rank == 0 && warp == 2 && lane == 0) atomicAdd(p.stall + 3, (unsigned long long)(clock64() - t_wait));
    tc_fence_before();
    __syncthreads();
    if (p.x_overlap) cluster_sync_all();   // every CTA's MMAs have completed (or it has given up): the rings may be written by the others
    if (abort_flag) {
        // A wait gave up: let the bulk copies counted on this CTA's barriers land and its MMAs retire before it goes on.  (Results are
        // unspecified now; every write still stays inside the cluster's exchange areas and the output.)
        if (warp == 0 && rank == 0)
            for (int back = 0; back < S && back < issued; ++back) {
                const int it = issued - 1 - back;
                for (uint32_t i = 0; i < kSkDrainPolls && !__all_sync(0xffffffffu, mbar_try_wait(&full_bar[it % S], (uint32_t)(it / S) & 1u)); ++i) {}
            }
        if (warp == 1 && rank == 0) {
            if (elect_one()) {
                if constexpr (PAIR) umma_commit_pair(&drain_bar, (uint16_t)(1u << leader));
                else umma_commit(&drain_bar);
            }
            __syncwarp();
            for (uint32_t i = 0; i < kSkDrainPolls && !__all_sync(0xffffffffu, mbar_try_wait(&drain_bar, 0u)); ++i) {}
        }
        __syncthreads();
    }
    tc_fence_after();

    const bool exchange = p.splits > 1 && k_total > 0;
    if (exchange) {
        // partial sums of the other CTAs' columns -> their exchange areas: block (sender, four columns) = 128 rows x 16 bytes; the next columns
        // are read from TMEM while the current ones are sent
        const int n8 = sw >> 3, c_lo = half ? (n8 + 1) >> 1 : 0, n_c = (half ? n8 : (n8 + 1) >> 1) - c_lo, n_all = n_c * (p.splits - 1);
        int f_dst = split + 1 < p.splits ? split + 1 : 0, f_ch = 0, s_dst = f_dst, s_ch = 0;   // next columns to read, next to send
        auto step = [&](int& dst, int& ch) {
            if (++ch == n_c) {
                ch = 0;
                if (++dst == p.splits) dst = 0;
            }
        };
        auto send = [&](const uint32_t (&r)[8]) {
            const uint32_t at = map_to_cta(smem_u32(ring) + (uint32_t)p.x_off + (uint32_t)(((split < s_dst ? split : split - 1) * (sw >> 2) + 2 * (c_lo + s_ch)) * 128 + m) * 16u,
                                           (uint32_t)(PAIR ? 2 * s_dst + rank : s_dst));
            st_cluster_v4(at, __uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
            st_cluster_v4(at + 2048u, __uint_as_float(r[4]), __uint_as_float(r[5]), __uint_as_float(r[6]), __uint_as_float(r[7]));
            step(s_dst, s_ch);
        };
        auto fetch = [&](uint32_t (&r)[8]) {
            tmem_ld8(t_row + (uint32_t)(f_dst * sw + (c_lo + f_ch) * 8), r);
            step(f_dst, f_ch);
        };
        if (n_all > 0) {
            uint32_t r0[8], r1[8];
            fetch(r0);
            tmem_ld_wait();
            for (int i = 0; i < n_all; i += 2) {
                if (i + 1 < n_all) fetch(r1);
                send(r0);
                if (i + 1 < n_all) {
                    tmem_ld_wait();
                    if (i + 2 < n_all) fetch(r0);
                    send(r1);
                    if (i + 2 < n_all) tmem_ld_wait();
                }
            }
        }
    }
    if (clustered) cluster_sync_all();   // the partial sums have arrived; nobody reads or writes another CTA's memory after this

    const bool do_stats = p.stats != nullptr;
    auto fetch = [&](uint32_t (&r)[16], int g) {
        uint32_t lo[8], hi[8];
        tmem_ld8(t_row + (uint32_t)(col0 + g * 16), lo);
        if (g * 16 + 16 <= sw) tmem_ld8(t_row + (uint32_t)(col0 + g * 16 + 8), hi);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            r[i] = lo[i];
            r[8 + i] = g * 16 + 16 <= sw ? hi[i] : 0u;
        }
    };
    const float4* xin = reinterpret_cast<const float4*>(ring + p.x_off) + m;
    const int x_sender = (sw >> 2) * 128;   // float4s of one sender
    for (int g = g_lo; g < g_hi; ++g) {
        const bool wide = g * 16 + 16 <= sw;
        uint32_t r[16];
        if (k_total > 0) {
            fetch(r, g);
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = 0u;
        }
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
        if (exchange) {
            const float4* in = xin + (size_t)4 * g * 128;
#pragma unroll 2
            for (int src = 1; src < p.splits; ++src, in += x_sender) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i < 2 || wide) {
                        const float4 f = in[i * 128];
                        v[4 * i] += f.x;
                        v[4 * i + 1] += f.y;
                        v[4 * i + 2] += f.z;
                        v[4 * i + 3] += f.w;
                    }
                }
            }
        }
        const int ch0 = c.ktile * p.n_tile + col0 + g * 16;
        if (p.bias != nullptr) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < 8 || wide) v[i] += __ldg(p.bias + ch0 + i);
        }
        if (p.out_is_f32) {
            if (row_valid) {
                float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + row_off + ch0);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < 2 || wide) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            continue;
        }
        uint32_t pk[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pk[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
        if (row_valid) {
            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.out) + row_off + ch0;
            if (p.out_v8 && wide && (ch0 & 15) == 0) {
                st_global_v8(dst, pk);
            } else {
                *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                if (wide) *reinterpret_cast<uint4*>(dst + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
        }
        if (do_stats) {   // sums of the values as stored
            if (!row_valid) {
#pragma unroll
                for (int i = 0; i < 8; ++i) pk[i] = 0u;
            }
            if constexpr (BWD) {
                float a[16], b[16];   // dz and dz * y of this row
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const f32x2 dz = bwd_pair(pk[4 * h + k], word_of(in[h].other, k), in[h].mask, k);
                        const float2 s = split_f32x2(dz), sy = split_f32x2(mul_f32x2(dz, widen_bf16x2(word_of(in[h].y, k))));
                        a[8 * h + 2 * k] = s.x; a[8 * h + 2 * k + 1] = s.y;
                        b[8 * h + 2 * k] = sy.x; b[8 * h + 2 * k + 1] = sy.y;
                    }
                if (g + 1 < g_hi) load_bwd(g + 1);
                butterfly16(a, b, lane);
                if ((lane & 1) == 0) {
                    s_sum[q][0][g * 16 + (lane >> 1)] = a[0];
                    s_sum[q][1][g * 16 + (lane >> 1)] = b[0];
                }
            } else {
                s_sum[q][total_is_square(lane)][g * 16 + column_of_total(lane)] = column_sums(pk, s_stage[warp], lane);
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (do_stats) {
        const int grp = p.stats_group_images > 0 ? c.n0 / p.stats_group_images : 0;
        double* st = p.stats + (size_t)grp * 2 * p.oc_valid + c.ktile * p.n_tile + col0;
        if (c.n0 < p.n_valid)   // (the second tile of a pair may lie past the last image)
            for (int i = threadIdx.x; i < sw; i += kSkThreads) {
                double s = 0.0, sq = 0.0;
                for (int w = 0; w < 4; ++w) {   // the four lane quarters
                    s += (double)s_sum[w][0][i];
                    sq += (double)s_sum[w][1][i];
                }
                atomicAdd(st + i, s);
                atomicAdd(st + p.oc_valid + i, sq);
            }
        __syncwarp();
    }
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, (uint32_t)p.tmem_cols);
        else tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
    if (TIMED && rank == 0 && threadIdx.x == 0) atomicAdd(p.stall + 4, (unsigned long long)(clock64() - t_start));
    pdl_end(p.no_wait);
    if constexpr (PAIR) cluster_sync_all();   // a pair gives its TMEM back together
}

static b2c_status splitk_optin(b2c_ctx* ctx)
{
    if (!(ctx->smem_optin_done & B2C_OPTIN_SPLITK)) {
        for (auto* k : {conv_splitk_kernel<false, false, false>, conv_splitk_kernel<false, true, false>, conv_splitk_kernel<true, false, false>, conv_splitk_kernel<true, true, false>,
                        conv_splitk_kernel<false, false, true>, conv_splitk_kernel<false, true, true>, conv_splitk_kernel<true, false, true>, conv_splitk_kernel<true, true, true>})
            B2C_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 210 * 1024));
        ctx->smem_optin_done |= B2C_OPTIN_SPLITK;
    }
    return B2C_OK;
}

int splitk_max_clusters(b2c_ctx* ctx, int cluster, bool pair)
{
    if (cluster == 1) return ctx->sm_count;
    int& known = ctx->max_clusters[pair ? 1 : 0][cluster];   // a property of the device: asked once per context
    if (known < 0) {
        known = 0;
        if (splitk_optin(ctx) != B2C_OK) return 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cluster);
        cfg.blockDim = dim3(kSkThreads);
        cfg.dynamicSmemBytes = 209 * 1024;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, pair ? conv_splitk_kernel<true, false, false> : conv_splitk_kernel<false, false, false>, &cfg) == cudaSuccess) known = n;
    }
    return known;
}

b2c_status launch_conv_splitk(b2c_ctx* ctx, const ConvKParams& p, int grid, size_t smem_bytes, cudaStream_t stream)
{
    b2c_status st = splitk_optin(ctx);
    if (st != B2C_OK) return st;
    const unsigned cluster = (unsigned)(p.splits * (p.pair ? 2 : 1));
    const bool timed = p.stall != nullptr;
    const bool bwd = p.bwd_y != nullptr;
    auto* kernel = p.pair ? (timed ? (bwd ? conv_splitk_kernel<true, true, true> : conv_splitk_kernel<true, true, false>)
                                   : (bwd ? conv_splitk_kernel<true, false, true> : conv_splitk_kernel<true, false, false>))
                          : (timed ? (bwd ? conv_splitk_kernel<false, true, true> : conv_splitk_kernel<false, true, false>)
                                   : (bwd ? conv_splitk_kernel<false, false, true> : conv_splitk_kernel<false, false, false>));
    B2C_CUDA(b2c_launch(ctx, kernel, dim3((unsigned)grid), dim3(kSkThreads), smem_bytes, stream, cluster, p));
    B2C_CUDA(cudaGetLastError());
    return B2C_OK;
}

}  // namespace b2c
