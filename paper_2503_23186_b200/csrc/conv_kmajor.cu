// Implicit-GEMM convolution with K-major operands on tcgen05: forward pass and data gradient.
//
//   D[128 pixels x n_tile channels] = sum over (tap, channel block) A[128 x kb] * B[n_tile x kb]^T
//
// A is an im2col tile staged by TMA: a 4-D box (kb channels, bw x bh pixels, bn images) of the
// gathered activation tensor, shifted by the tap's offset; rows that fall outside the image are
// zero-filled by the TMA unit, which implements the padding.  Stride-2 forward convolutions
// gather from four "parity views" of the input (even/odd rows x even/odd columns), each a plain
// strided tensor map; the stride-2 data gradient is four sub-problems, one per output parity.
// B is a box (kb channels, one tap, n_tile output channels) of the [out][tap][in] weights.
//
// The kernel is persistent: one CTA per SM walks a list of (pixel tile, channel tile) units.
//   * Two or four accumulators in TMEM (four where 4 x n_tile columns fit): while the epilogue warps drain unit i
//     (bias, bf16 rounding, BatchNorm sums, stores), the MMA threads already accumulate the next units into the
//     others, and the TMA producers run ahead through the shared-memory ring across unit boundaries.
//   * Vertical tap reuse (3x3, stride 1, tile inside one image): a stage holds the tile plus one
//     halo row above and below for one horizontal shift; the three vertical taps read it at row
//     offsets of one image row (a multiple of the swizzle period), so the input is fetched three
//     times instead of nine.
//   * Small filter banks stay resident in shared memory for the whole launch.
// Warp roles: warp 0 = first TMA producer, warp 1 = TMEM owner + first MMA issuer, warps 2..9 = epilogue (two per TMEM
// lane quarter, splitting the columns), warp 10 = second MMA issuer (the two issuers take alternate units), warp 11 = second
// TMA producer (the two producers take alternate stages).  Producer and issuer warps run their loops with all lanes and issue
// from one elected lane.  Every mbarrier wait is bounded.
#include "conv_kmajor.h"

namespace b2c {

static constexpr int kMaxStages = 8;   // (conv_splitk.cu has room for as many)
static constexpr int kMaxAccBufs = 4;
static constexpr int kEpiWarps = 8;
static constexpr int kIssuers = 2;       // MMA-issuing threads: warp 1 and the warps after the epilogue warps
static constexpr int kProducers = 2;     // TMA-issuing threads: warp 0 and the warp after the issuer warps; they take alternate stages
static constexpr int kThreads = 64 + 32 * kEpiWarps + 32 * (kIssuers - 1) + 32 * (kProducers - 1);
static constexpr int kProducerWarp1 = 2 + kEpiWarps + (kIssuers - 1);   // warp index of the second producer
static constexpr uint32_t kDrainPolls = 1u << 22;
static constexpr size_t kClusterSmem = 115 * 1024;   // more than half of the 228 KB of an SM
static constexpr int kFoldUnits = 8;     // units of a narrow tile (wide: half as many) whose squares a lane of the epilogue adds up before they move on

// Units of this CTA (a CTA pair walks pair-units: two pixel tiles next to each other, same channel tile, of which CTA `rank` takes tile
// 2*m + rank).  A walker keeps its channel tile.  The walkers take their units in turns, so that tiles in work at one time are neighbours in
// memory; where a pass sums several statistics groups, each takes a run of consecutive pixel tiles instead, so that it meets at most two
// groups or so: in turns, every walker met every group, and all of them sent the group's sums to the same addresses at the same time.  Eight
// groups of 128 images: ResNet-18-shaped step 5853 -> 5555 us (launch times summed), ResNet-50-shaped 24.49 -> 23.70 ms.  Without groups runs
// are slower: data gradient 112 <- 256 1x1 at 32x32 with 442 images 79.3 us in runs, 72.5 in turns, 64 <- 256 with 1024 images 104.0 and 102.7.
struct UnitWalk {
    int first, stride, count, rank, pair;
    __device__ UnitWalk(const ConvKParams& p, int rank_) : rank(rank_), pair(p.pair)
    {
        const int w = pair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, walkers = pair ? (int)(gridDim.x >> 1) : (int)gridDim.x;
        count = pair ? p.total_units >> 1 : p.total_units;
        first = w;
        stride = walkers;
        if (p.stats != nullptr && p.stats_group_images > 0) {
            const int per_ktile = walkers / p.n_ktiles, j = w / p.n_ktiles, kt = w - j * p.n_ktiles, m = count / p.n_ktiles;   // (walkers is a multiple of n_ktiles)
            first = (int)((long long)m * j / per_ktile) * p.n_ktiles + kt;
            count = (int)((long long)m * (j + 1) / per_ktile) * p.n_ktiles;
            stride = p.n_ktiles;
        }
    }
    __device__ int unit(const ConvKParams& p, int pu) const
    {
        return pair ? (2 * (pu / p.n_ktiles) + rank) * p.n_ktiles + pu % p.n_ktiles : pu;
    }
};
__device__ __forceinline__ int unit_iters(const ConvKParams& p, int par)
{
    const int taps = p.taps[par].count;
    if (p.fh || p.hm) return p.c_blocks;
    return (p.vreuse ? taps / 3 : taps) * p.c_blocks;
}

// ring slots a unit takes: gsub k-blocks per slot, the last slot of a unit possibly with fewer
__device__ __forceinline__ int unit_stages(const ConvKParams& p, int par)
{
    const int n = unit_iters(p, par);
    return p.gsub > 1 ? (n + p.gsub - 1) / p.gsub : n;
}

// Epilogue of one warp over all units of the CTA, for the tile widths and plans that epilogue_blocks does not take (up to 48 channels, 80 to 112,
// 144 to 240; rings that leave no room; a bias or fp32 output).  Epilogue warp e reads the TMEM lane quarter its warp index selects and the column
// half e >> 2 of every accumulator.  The warp owns at most NCH 16-column chunks per unit.  EAGER: it reads all
// its columns at once and hands the accumulator back before packing and storing (narrow tiles).
// STATS: BatchNorm sums of the values as stored, kept in registers until the statistics group ends; those of the last group are left
// in my_stats ([0, 128) sums, [128, 256) sums of squares) for the CTA to add up.  Returns that group and channel tile (-1: none).
//   * EAGER: a lane sums its own row's columns (32 registers per chunk), a butterfly reduces over the rows once per group.
//   * wide tiles: two exchanges between lanes first (add_chunk), a quarter of the registers and about 65 instructions per chunk.
//     Bound: issue slots and latency of eight warps.  Measured with 1024 images, forward with sums, on layers that have since gone to the blocks,
//     128 -> 128 at 16x16 and 1x1 64 -> 256 at 32x32: shuffle butterfly per chunk (150 instructions) 82 and 342 us; tensor cores (m16n8k16, which queue behind the
//     convolution's own MMAs) 90 and 224; transposed through shared memory (two warp barriers and a chain of eight adds) 72 and 253;
//     read from TMEM once more in the fragment layout 72 and 244; this 72 and 273 us (a rolled loop: 79 and 219).
// The squares of bf16 values end in the same few bits: added one by one to a running fp32 sum they are rounded down more often than up,
// and a chain of 200 comes out 5e-7 low.  So four squares of a wide tile meet before they reach the running sum, which moves on to a second
// one in local memory after every few units; narrow tiles, which have no registers to spare, add their rows up in my_stats instead.
// Sums of squares of 1024 images are 1.2e-8 off (measured on the same layers, without it: 3.3e-7 on 64 -> 256 1x1, 4.6e-8 on 32 -> 64 1x1; with it 1.2e-8 too on 16 -> 32 1x1, 1.3e-8 on 160 -> 160 and 64 -> 256 3x3),
// for 275 -> 280 us on 64 -> 256 1x1, 64.9 -> 66.1 on 128 -> 128 at 16x16, 76.6 -> 80.8 on 64 -> 64 at 32x32.
// Without STATS the code carries no accumulators: 1x1 64 -> 256 154 -> 126 us, 32 -> 64 57 -> 48 us, data gradient 256 -> 64 159 -> 132 us.
template <int NCH, bool EAGER, bool HM, bool STATS>
__device__ __forceinline__ int2 epilogue_loop(const ConvKParams& p, uint32_t tmem_base, uint64_t* acc_full, uint64_t* acc_empty,
                                              uint32_t* abort_flag, float* my_stats, int e, int lane, int rank)
{
    const UnitWalk walk(p, rank);
    // the accumulator-free barrier lives in the leader CTA of a pair: the peer's warps arrive on it remotely
    const bool remote_empty = p.pair && rank != 0;
    const int q = (e + 2) & 3;       // TMEM lane quarter this warp may read: (warp index in the CTA) % 4, epilogue warps start at 2
    const int m = q * 32 + lane;     // accumulator row = pixel of the tile (w fastest, then h, then image)
    const int lw = m % p.bw, lh = (m / p.bw) % p.bh, ln = m / (p.bw * p.bh);
    const int n_chunks_all = p.n_tile >> 4;
    const int first_half = (n_chunks_all + 1) >> 1;
    const int ck_begin = (e >> 2) ? first_half : 0;
    const int n_chunks = (e >> 2) ? n_chunks_all - first_half : first_half;   // chunks this warp handles
    const int col_begin = ck_begin * 16;
    constexpr int NA = !STATS ? 1 : EAGER ? 8 * NCH : 2 * NCH;   // column pairs this lane sums
    f32x2 acc_s[NA], acc_q[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) acc_s[i] = acc_q[i] = 0ull;
    f32x2 long_q[NA];   // wide tiles only
    int opaque_zero = 0, held = 0;   // (an index that the compiler cannot see through keeps long_q out of the registers)
    if constexpr (STATS && !EAGER) {
        asm volatile("mov.u32 %0, 0;" : "=r"(opaque_zero));
#pragma unroll
        for (int i = 0; i < NA; ++i) long_q[i + opaque_zero] = 0ull;
    }
    if constexpr (STATS && EAGER) {
        for (int i = lane; i < 256; i += 32) my_stats[i] = 0.f;
        __syncwarp();
    }
    int jacc = 0, cur_group = -1, cur_ktile = 0;
    bool ok = true;
    long long epi_wait = 0;

    // Totals over the warp's 32 rows: emit(column of the warp, sum, sum of squares) in one lane per column.
    auto each_total = [&](auto emit) {
        if constexpr (STATS && EAGER) {
#pragma unroll
            for (int ck = 0; ck < NCH; ++ck) {
                float a[16], b[16];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 s = split_f32x2(acc_s[ck * 8 + i]), sq = split_f32x2(acc_q[ck * 8 + i]);
                    a[2 * i] = s.x; a[2 * i + 1] = s.y;
                    b[2 * i] = sq.x; b[2 * i + 1] = sq.y;
                }
                butterfly16(a, b, lane);
                if ((lane & 1) == 0 && ck < n_chunks) emit(ck * 16 + (lane >> 1), a[0], b[0]);
            }
        } else if constexpr (STATS) {
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const float2 s = column_total(acc_s[i]), sq = column_total(add_f32x2(acc_q[i], long_q[i + opaque_zero]));
                if ((lane & 7) == 0 && i < 2 * n_chunks) {
                    const int col = (i >> 1) * 16 + column_of(lane) + 2 * (i & 1);
                    emit(col, s.x, sq.x);
                    emit(col + 1, s.y, sq.y);
                }
            }
        }
        __syncwarp();
    };
    // The running sums move on; at the end of a statistics group this warp's share of it goes to global fp64.
    auto flush_stats = [&](bool group_done) {
        held = 0;
        double* st = p.stats + (size_t)cur_group * 2 * p.oc_valid + cur_ktile * p.n_tile + col_begin;
        if constexpr (EAGER) {
            each_total([&](int col, float s, float sq) {   // (a column's total always comes from the same lane)
                my_stats[col] += s;
                my_stats[128 + col] += sq;
            });
            if (group_done) {
                for (int col = lane; col < n_chunks * 16; col += 32) {
                    atomicAdd(st + col, (double)my_stats[col]);
                    atomicAdd(st + p.oc_valid + col, (double)my_stats[128 + col]);
                    my_stats[col] = my_stats[128 + col] = 0.f;
                }
                __syncwarp();
            }
#pragma unroll
            for (int i = 0; i < NA; ++i) acc_s[i] = acc_q[i] = 0ull;
        } else {
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                long_q[i + opaque_zero] = add_f32x2(long_q[i + opaque_zero], acc_q[i]);
                acc_q[i] = 0ull;
            }
            if (group_done) {
                each_total([&](int col, float s, float sq) {
                    atomicAdd(st + col, (double)s);
                    atomicAdd(st + p.oc_valid + col, (double)sq);
                });
#pragma unroll
                for (int i = 0; i < NA; ++i) acc_s[i] = long_q[i + opaque_zero] = 0ull;
            }
        }
    };

    // The coordinates of a unit are worked out one unit ahead, between the probe of the current unit's accumulator barrier
    // and the use of its answer: the barrier's latency and the integer chain of the decode (about 350 cycles each, measured)
    // run side by side instead of one after the other.
    UnitCoord c_next = decode_unit(p, walk.unit(p, walk.first < walk.count ? walk.first : 0));
    for (int pu = walk.first; pu < walk.count; pu += walk.stride) {
        const UnitCoord c = c_next;
        const int n_it = unit_iters(p, c.par);
        int buf = 0;
        uint32_t full_now = 0;
        if (n_it > 0) {
            buf = jacc & (p.acc_bufs - 1);
            full_now = mbar_try_wait(&acc_full[buf], (uint32_t)(jacc >> p.acc_shift) & 1u) ? 1u : 0u;   // all lanes, one address
        }
        if (pu + walk.stride < walk.count) c_next = decode_unit(p, walk.unit(p, pu + walk.stride));
        const bool row_valid = (c.n0 + ln) < p.n_valid;
        const long long row_off = (long long)(c.n0 + ln) * p.os_n + (long long)(c.oh0 + lh) * p.os_h + (long long)(c.ow0 + lw) * p.os_w + p.off[c.par];
        if (n_it > 0) {
            if (!__all_sync(0xffffffffu, full_now != 0u)) {   // not full yet: one poller per warp
                const long long w3 = clock64();
                ok = true;
                if (lane == 0) ok = mbar_wait_bounded(&acc_full[buf], (uint32_t)(jacc >> p.acc_shift) & 1u, p.spin_limit, abort_flag);
                epi_wait += clock64() - w3;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) atomicOr(p.status, B2C_DEV_TIMEOUT);
                    break;
                }
            }
            tc_fence_after();
            ++jacc;
        }
        // A new statistics group: the finished group's sums go out, after this unit's first columns have been read (narrow tiles: after its
        // accumulator has been handed back), so that the MMA threads do not wait for it.
        bool flush_pending = false;
        int next_group = cur_group;
        if constexpr (STATS) {
            next_group = p.stats_group_images > 0 ? (p.grp_shift >= 0 ? c.n0 >> p.grp_shift : c.n0 / p.stats_group_images) : 0;
            flush_pending = cur_group >= 0 && (next_group != cur_group || held == (EAGER ? kFoldUnits : kFoldUnits / 2));
        }
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * p.acc_cols + col_begin);
        // the accumulator is handed back to the MMA thread as soon as this warp has read its last column
        auto release = [&]() {
            if (n_it > 0) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (remote_empty) mbar_arrive_cluster(map_to_cta(smem_u32(&acc_empty[buf]), 0));
                    else mbar_arrive(&acc_empty[buf]);
                }
            }
        };
        // bias, rounding and stores of one 16-column chunk; returns the values as stored in pk
        auto store_chunk = [&](const uint32_t (&r)[16], int c0, uint32_t (&pk)[8]) {
            const int ch0 = c.ktile * p.n_tile + col_begin + c0;  // first output channel of this chunk
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
            if (!HM && p.bias != nullptr) {   // (merged-tap plans have neither a bias nor fp32 output)
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] += (ch0 + i < p.oc_valid) ? __ldg(p.bias + ch0 + i) : 0.f;
            }
            if (!HM && !STATS && p.out_is_f32) {   // (statistics are those of bf16 values)
                if (row_valid) {
                    float* dst = reinterpret_cast<float*>(p.out) + row_off + ch0;
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        if (ch0 + i < p.oc_valid) *reinterpret_cast<float4*>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                }
                return;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) pk[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
            if (row_valid) {
                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.out) + row_off + ch0;
                if (p.out_v8 && ch0 + 8 < p.oc_valid) {
                    st_global_v8(dst, pk);   // one full 32-byte sector per lane
                } else {
                    if (ch0 < p.oc_valid) *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    if (ch0 + 8 < p.oc_valid) *reinterpret_cast<uint4*>(dst + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                }
            }
        };

        auto group_end = [&]() {
            if constexpr (!STATS) return;
            if (flush_pending) flush_stats(next_group != cur_group);   // still the previous units' sums, group and channel tile
            ++held;
            cur_group = next_group;
            cur_ktile = c.ktile;
        };
        if constexpr (EAGER) {
            // narrow tiles: read all of this warp's columns at once, free the accumulator, then work from registers
            uint32_t r[NCH][16];
            if constexpr (HM) {
                // Merged horizontal taps: the accumulator holds three blocks of n_tile columns, block s = the contribution of
                // filter column s evaluated at this row's own pixel.  Output pixel w takes block 0 of pixel w - 1, block 1 of its
                // own pixel and block 2 of pixel w + 1; a warp's 32 rows are whole image rows, so the neighbours are the
                // adjacent lanes, and the first / last pixel of an image row has no left / right neighbour (zero padding).
                const float m_left = lw != 0 ? 1.f : 0.f, m_right = lw != p.bw - 1 ? 1.f : 0.f;
#pragma unroll
                for (int ck = 0; ck < NCH; ++ck) {
                    uint32_t d0[16], d1[16], d2[16];
                    tmem_ld16(t_row + (uint32_t)(ck * 16), d0);
                    tmem_ld16(t_row + (uint32_t)(p.n_tile + ck * 16), d1);
                    tmem_ld16(t_row + (uint32_t)(2 * p.n_tile + ck * 16), d2);
                    tmem_ld_wait();
                    if (ck == NCH - 1) release();
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float left = __shfl_up_sync(0xffffffffu, __uint_as_float(d0[i]), 1);
                        const float right = __shfl_down_sync(0xffffffffu, __uint_as_float(d2[i]), 1);
                        r[ck][i] = __float_as_uint(fmaf(left, m_left, fmaf(right, m_right, __uint_as_float(d1[i]))));
                    }
                }
            } else {
#pragma unroll
                for (int ck = 0; ck < NCH; ++ck) {
                    if (n_it > 0 && ck < n_chunks) {
                        tmem_ld16(t_row + (uint32_t)(ck * 16), r[ck]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i) r[ck][i] = 0u;
                    }
                }
                if (n_it > 0) tmem_ld_wait();
                release();
            }
            group_end();
#pragma unroll
            for (int ck = 0; ck < NCH; ++ck) {
                if (ck < n_chunks) {
                    uint32_t pk[8];
                    store_chunk(r[ck], ck * 16, pk);
                    if (STATS && row_valid) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) add_pair(pk[i], acc_s[STATS ? ck * 8 + i : 0], acc_q[STATS ? ck * 8 + i : 0]);
                    }
                }
            }
        } else if constexpr (STATS) {
            // (only convolutions with taps everywhere have statistics: n_it > 0)
            uint32_t r[2][16];
            if (n_chunks > 0) {
                tmem_ld16(t_row, r[0]);
                tmem_ld_wait();
            }
            if (n_chunks <= 1) release();
            group_end();
#pragma unroll
            for (int ck = 0; ck < NCH; ++ck) {
                if (ck < n_chunks) {   // the next chunk comes in while this one is stored and summed
                    if (ck + 1 < n_chunks) tmem_ld16(t_row + (uint32_t)((ck + 1) * 16), r[(ck + 1) & 1]);
                    uint32_t pk[8];
                    store_chunk(r[ck & 1], ck * 16, pk);
                    if (!row_valid) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) pk[i] = 0u;
                    }
                    __syncwarp();
                    f32x2 s[2] = {acc_s[2 * ck], acc_s[2 * ck + 1]}, sq[2] = {acc_q[2 * ck], acc_q[2 * ck + 1]};
                    add_chunk(pk, lane, s, sq);
                    acc_s[2 * ck] = s[0]; acc_s[2 * ck + 1] = s[1];
                    acc_q[2 * ck] = sq[0]; acc_q[2 * ck + 1] = sq[1];
                    if (ck + 1 < n_chunks) {
                        tmem_ld_wait();
                        if (ck + 2 == n_chunks) release();
                    }
                }
            }
        } else {
            auto process = [&](const uint32_t (&r)[16], int c0) {
                uint32_t pk[8];
                store_chunk(r, c0, pk);
            };
            uint32_t ra[16], rb[16];
            if (n_it > 0 && n_chunks > 0) {
                tmem_ld16(t_row, ra);
                tmem_ld_wait();
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) ra[i] = rb[i] = 0u;
            }
            if (n_chunks <= 1) release();
            for (int ck = 0; ck < n_chunks; ck += 2) {
                // chunk ck is in ra; fetch ck+1 into rb while ra is processed, then ck+2 into ra while rb is processed
                if (n_it > 0 && ck + 1 < n_chunks) tmem_ld16(t_row + (uint32_t)((ck + 1) * 16), rb);
                process(ra, ck * 16);
                if (ck + 1 < n_chunks) {
                    if (n_it > 0) {
                        tmem_ld_wait();
                        if (ck + 2 == n_chunks) release();
                        if (ck + 2 < n_chunks) tmem_ld16(t_row + (uint32_t)((ck + 2) * 16), ra);
                    }
                    process(rb, (ck + 1) * 16);
                    if (n_it > 0 && ck + 2 < n_chunks) {
                        tmem_ld_wait();
                        if (ck + 3 == n_chunks) release();
                    }
                }
            }
        }
    }
    // the four lane quarters' sums meet in shared memory: a quarter of the global atomics at the kernel's end
    if (STATS && cur_group >= 0 && ok)
        each_total([&](int col, float s, float sq) {
            my_stats[col] = EAGER ? my_stats[col] + s : s;
            my_stats[128 + col] = EAGER ? my_stats[128 + col] + sq : sq;
        });
    if (p.stall != nullptr && e == 0 && lane == 0) atomicAdd(p.stall + 3, (unsigned long long)epi_wait);
    return STATS && ok ? make_int2(cur_group, cur_ktile) : make_int2(-1, 0);
}

// Epilogue of one warp for tiles of 64, 128 or 256 channels without a bias: the same share of every unit as in epilogue_loop, but the rounded
// values go through shared memory, BC columns of the warp's 32 rows at a time, so that a lane then holds 8 neighbouring columns of every
// (32 / (BC / 8))-th row: an instruction stores whole runs of BC columns (BC = 64: 4 lines, where a row per lane touches 32), and the
// BatchNorm sums of a column are additions in one lane with no exchange.  Rows that do not exist (images past the last one) are skipped.
// NB blocks of BC columns are the warp's half of the tile; wider blocks need fewer running sums per lane (with NB = 4 and BC = 32 they spill).
// Bound: HBM writes on 1x1 layers (537 MB alone take 125-145 us), else the two warps' latency per scheduler, no longer the store path.
// Layers of 1024 images inside a step, epilogue_loop -> this: with sums 64 -> 256 1x1 at 32x32 312 -> 145 us (sums in a pass of their own: 139 +
// 95), 128 -> 512 at 16x16 166 -> 84, 64 -> 64 3x3 80 -> 71, 128 -> 128 3x3 at 16x16 77 -> 63, 64 -> 128 1x1 stride 2 60 -> 41, 512 -> 512 at 4x4
// 65 -> 63; without sums data gradient 256 <- 64 1x1 137 -> 126, 512 <- 128 81 -> 71, 64 <- 64 3x3 66 -> 63.
// Every four units the running squares move on to a second sum in local memory, and what that addition rounds off stays behind (not with blocks
// of 16 columns, where the sixteen pairs' extra instructions and spills cost 128 -> 128 at 16x16 66.9 -> 74.7 us inside a step): squares of positive outputs of 2048 images (16 -> 64 1x1) are 2.1e-9 off, 4.3e-8 without the remainder, of 1024 images (128 -> 512 1x1) 7.9e-9 and 1.0e-8.
// Tiles of 64 channels have registers for a second plain sum too (16 -> 64 1x1 with 1024 images 49.7 -> 50.6 us for both); wider ones keep
// one for the whole statistics group, as in epilogue_loop: sums of 1024 images with a mean are 0.2-1.4e-9 of their magnitudes off, there and here.
template <int BC, int NB, bool HM, bool STATS>
__device__ __forceinline__ int2 epilogue_blocks(const ConvKParams& p, uint32_t tmem_base, uint64_t* acc_full, uint64_t* acc_empty, uint32_t* abort_flag,
                                                float* my_stats, uint8_t* stage, int e, int lane, int rank)
{
    constexpr int LPR = BC / 8;       // lanes per row on the way out
    constexpr int RPI = 32 / LPR;     // rows per instruction; LPR instructions cover the warp's rows
    const UnitWalk walk(p, rank);
    const bool remote_empty = p.pair && rank != 0;
    const int q = (e + 2) & 3;
    const int col_begin = (e >> 2) * (BC * NB);
    const int my_row = q * 32 + lane / LPR;   // and every RPI-th after it
    int my_off = 8 * (lane % LPR) + col_begin;
#pragma unroll
    for (int bit = 0; bit < 7; ++bit)
        if ((my_row >> bit) & 1) my_off += p.row_bit[bit];
    constexpr int LOG_RPI = RPI == 4 ? 2 : RPI == 8 ? 3 : 4;
    int step_off[5 - LOG_RPI];   // (moved by hand: read from the parameters again for every store, they cost 64 -> 64 3x3 with 256 images 18.2 -> 19.2 us)
#pragma unroll
    for (int i = 0; i < 5 - LOG_RPI; ++i) asm volatile("mov.u32 %0, %1;" : "=r"(step_off[i]) : "r"(p.row_bit[LOG_RPI + i]));
    // 16-byte words of the staging block: word j of row r lies at j ^ swizzle(r), without bank conflicts either way
    auto swizzle = [](int row) { return BC == 64 ? row & 7 : BC == 32 ? (row >> 1) & 3 : (row >> 2) & 1; };
    const uint32_t st_w = smem_u32(stage) + (uint32_t)lane * (BC * 2);
    const int sw_w = swizzle(lane);

    constexpr int NA = STATS ? 4 * NB : 1;   // column pairs this lane sums
    constexpr bool LONG_S = STATS && BC == 32;   // tiles of 64 channels have registers for a second running sum
    f32x2 acc_s[NA], acc_q[NA], long_s[LONG_S ? NA : 1], long_q[NA];
    int opaque_zero = 0, held = 0;   // (an index that the compiler cannot see through keeps long_q out of the registers)
    if constexpr (STATS) {
        asm volatile("mov.u32 %0, 0;" : "=r"(opaque_zero));
#pragma unroll
        for (int i = 0; i < NA; ++i) acc_s[i] = acc_q[i] = long_q[i + opaque_zero] = 0ull;
#pragma unroll
        for (int i = 0; i < (LONG_S ? NA : 1); ++i) long_s[i] = 0ull;
    }
    int jacc = 0, cur_group = -1, cur_ktile = 0;
    bool ok = true;
    long long epi_wait = 0;

    auto each_total = [&](auto emit) {   // emit(column of the warp, sum, sum of squares) in one lane per column
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            float2 s = split_f32x2(LONG_S ? add_f32x2(acc_s[i], long_s[LONG_S ? i : 0]) : acc_s[i]), sq = split_f32x2(add_f32x2(acc_q[i], long_q[i + opaque_zero]));
#pragma unroll
            for (int bit = LPR; bit < 32; bit <<= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, bit);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, bit);
                sq.x += __shfl_xor_sync(0xffffffffu, sq.x, bit);
                sq.y += __shfl_xor_sync(0xffffffffu, sq.y, bit);
            }
            if (lane < LPR) {
                const int col = (i >> 2) * BC + 8 * lane + 2 * (i & 3);
                emit(col, s.x, sq.x);
                emit(col + 1, s.y, sq.y);
            }
        }
        __syncwarp();
    };
    auto flush_stats = [&](bool group_done) {
        held = 0;
        const f32x2 minus_one = make_f32x2(-1.f, -1.f);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const f32x2 old_q = long_q[i + opaque_zero], new_q = add_f32x2(old_q, acc_q[i]);
            long_q[i + opaque_zero] = new_q;
            if constexpr (BC != 16) acc_q[i] = add_f32x2(acc_q[i], fma_f32x2(new_q, minus_one, old_q));   // what the addition rounds off stays behind
            else acc_q[i] = 0ull;
            if constexpr (LONG_S) {
                long_s[i] = add_f32x2(long_s[i], acc_s[i]);
                acc_s[i] = 0ull;
            }
        }
        if (group_done) {
            double* st = p.stats + (size_t)cur_group * 2 * p.oc_valid + cur_ktile * p.n_tile + col_begin;
            each_total([&](int col, float s, float sq) {
                atomicAdd(st + col, (double)s);
                atomicAdd(st + p.oc_valid + col, (double)sq);
            });
#pragma unroll
            for (int i = 0; i < NA; ++i) acc_s[i] = acc_q[i] = long_q[i + opaque_zero] = 0ull;
#pragma unroll
            for (int i = 0; i < (LONG_S ? NA : 1); ++i) long_s[i] = 0ull;
        }
    };

    const int m_lane = q * 32 + lane, lw = m_lane & (p.bw - 1);   // (merged taps: position in the image row)
    const float m_left = lw != 0 ? 1.f : 0.f, m_right = lw != p.bw - 1 ? 1.f : 0.f;
    // (the next unit's coordinates are worked out while the barrier is probed, as in epilogue_loop)
    UnitCoord c_next = decode_unit(p, walk.unit(p, walk.first < walk.count ? walk.first : 0));
    for (int pu = walk.first; pu < walk.count; pu += walk.stride) {
        const UnitCoord c = c_next;
        const int n_it = unit_iters(p, c.par);
        int buf = 0;
        uint32_t full_now = 0;
        if (n_it > 0) {
            buf = jacc & (p.acc_bufs - 1);
            full_now = mbar_try_wait(&acc_full[buf], (uint32_t)(jacc >> p.acc_shift) & 1u) ? 1u : 0u;
        }
        if (pu + walk.stride < walk.count) c_next = decode_unit(p, walk.unit(p, pu + walk.stride));
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + ((long long)c.n0 * p.os_n + (long long)c.oh0 * p.os_h + (long long)c.ow0 * p.os_w +
                             p.off[c.par] + c.ktile * p.n_tile + my_off);
        const int images = p.n_valid - c.n0;   // (the second tile of a pair may lie past the last image)
        const int rows = images >= p.bn ? 128 : images > 0 ? images * p.bw * p.bh : 0;
        if (n_it > 0) {
            if (!__all_sync(0xffffffffu, full_now != 0u)) {
                const long long w3 = clock64();
                ok = true;
                if (lane == 0) ok = mbar_wait_bounded(&acc_full[buf], (uint32_t)(jacc >> p.acc_shift) & 1u, p.spin_limit, abort_flag);
                epi_wait += clock64() - w3;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) atomicOr(p.status, B2C_DEV_TIMEOUT);
                    break;
                }
            }
            tc_fence_after();
            ++jacc;
        }
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * p.acc_cols + col_begin);
        auto release = [&]() {
            if (n_it > 0) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (remote_empty) mbar_arrive_cluster(map_to_cta(smem_u32(&acc_empty[buf]), 0));
                    else mbar_arrive(&acc_empty[buf]);
                }
            }
        };
        uint32_t r[BC / 16][16];
        auto fetch = [&](int b) {
#pragma unroll
            for (int ck = 0; ck < BC / 16; ++ck) tmem_ld16(t_row + (uint32_t)(b * BC + ck * 16), r[ck]);
        };
        if constexpr (HM) {   // (see epilogue_loop; one block)
#pragma unroll
            for (int ck = 0; ck < BC / 16; ++ck) {
                uint32_t d0[16], d1[16], d2[16];
                tmem_ld16(t_row + (uint32_t)(ck * 16), d0);
                tmem_ld16(t_row + (uint32_t)(p.n_tile + ck * 16), d1);
                tmem_ld16(t_row + (uint32_t)(2 * p.n_tile + ck * 16), d2);
                tmem_ld_wait();
                if (ck == BC / 16 - 1) release();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float left = __shfl_up_sync(0xffffffffu, __uint_as_float(d0[i]), 1);
                    const float right = __shfl_down_sync(0xffffffffu, __uint_as_float(d2[i]), 1);
                    r[ck][i] = __float_as_uint(fmaf(left, m_left, fmaf(right, m_right, __uint_as_float(d1[i]))));
                }
            }
        } else if (n_it > 0) {
            fetch(0);
            tmem_ld_wait();
            if (NB == 1) release();
        } else {
#pragma unroll
            for (int ck = 0; ck < BC / 16; ++ck)
#pragma unroll
                for (int i = 0; i < 16; ++i) r[ck][i] = 0u;
        }
        if constexpr (STATS) {   // the previous units' sums
            const int next_group = p.stats_group_images > 0 ? (p.grp_shift >= 0 ? c.n0 >> p.grp_shift : c.n0 / p.stats_group_images) : 0;
            if (cur_group >= 0 && (next_group != cur_group || held == kFoldUnits / 2)) flush_stats(next_group != cur_group);
            ++held;
            cur_group = next_group;
            cur_ktile = c.ktile;
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            __syncwarp();   // the previous block has been read
#pragma unroll
            for (int j = 0; j < BC / 8; ++j) {
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int col = 8 * j + 2 * i;
                    w[i] = pack_bf16x2(__uint_as_float(r[col / 16][col % 16]), __uint_as_float(r[col / 16][col % 16 + 1]));
                }
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(st_w + 16u * (uint32_t)(j ^ sw_w)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
            }
            __syncwarp();
            if (b + 1 < NB && n_it > 0) fetch(b + 1);   // comes in while this block goes out
            constexpr int U = LPR < 4 ? LPR : 4;
#pragma unroll
            for (int i0 = 0; i0 < LPR; i0 += U) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int row = lane / LPR + RPI * (i0 + u);
                    const uint32_t at = smem_u32(stage) + (uint32_t)row * (BC * 2) + 16u * (uint32_t)((lane % LPR) ^ swizzle(row));
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w) : "r"(at) : "memory");
                    if (my_row + RPI * (i0 + u) < rows) {
                        int off = b * BC;
#pragma unroll
                        for (int t = 0; t < 5 - LOG_RPI; ++t)
                            if (((i0 + u) >> t) & 1) off += step_off[t];
                        *reinterpret_cast<uint4*>(out + off) = v[u];
                    } else {
                        v[u] = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
                if constexpr (STATS) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        f32x2 f[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) f[u] = widen_bf16x2(k == 0 ? v[u].x : k == 1 ? v[u].y : k == 2 ? v[u].z : v[u].w);
                        f32x2 s = add_f32x2(f[0], f[1]), sq = fma_f32x2(f[1], f[1], mul_f32x2(f[0], f[0]));
                        if constexpr (U == 4) {
                            s = add_f32x2(s, add_f32x2(f[2], f[3]));
                            sq = add_f32x2(sq, fma_f32x2(f[3], f[3], mul_f32x2(f[2], f[2])));
                        }
                        acc_s[4 * b + k] = add_f32x2(acc_s[4 * b + k], s);
                        acc_q[4 * b + k] = add_f32x2(acc_q[4 * b + k], sq);
                    }
                }
            }
            if (b + 1 < NB && n_it > 0) {
                tmem_ld_wait();
                if (b + 2 == NB) release();
            }
        }
    }
    if constexpr (STATS) asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");   // (blocks may lie where the sums go)
    if (STATS && cur_group >= 0 && ok)
        each_total([&](int col, float s, float sq) {
            my_stats[col] = s;
            my_stats[128 + col] = sq;
        });
    if (p.stall != nullptr && e == 0 && lane == 0) atomicAdd(p.stall + 3, (unsigned long long)epi_wait);
    return STATS && ok ? make_int2(cur_group, cur_ktile) : make_int2(-1, 0);
}

// Issues the MMAs of one stage: NB sub-tiles (vertical taps) x KS k-steps of 16 channels, fully unrolled so that
// the issuing thread spends a handful of independent instructions per MMA (its own dependent-issue latency, not the
// tensor pipe, bounds small-N tiles otherwise).  Descriptor low words advance by 32 bytes per k-step inside the
// swizzle atom and by a_step / b_step per sub-tile.
template <int KS, int NB, bool PAIR>
__device__ __forceinline__ void issue_stage(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                            uint32_t a_step16, uint32_t b_step16, uint32_t accumulate_first)
{
#pragma unroll
    for (int j = 0; j < NB; ++j) {
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const uint64_t ad = ((uint64_t)desc_hi << 32) | (uint64_t)(a_lo + (uint32_t)j * a_step16 + 2u * k);
            const uint64_t bd = ((uint64_t)desc_hi << 32) | (uint64_t)(b_lo + (uint32_t)j * b_step16 + 2u * k);
            if constexpr (PAIR) umma_bf16_pair(d_tmem, ad, bd, idesc, (j == 0 && k == 0) ? accumulate_first : 1u);
            else umma_bf16(d_tmem, ad, bd, idesc, (j == 0 && k == 0) ? accumulate_first : 1u);
        }
    }
}

// Full-halo stage: the A tile is a box of (bw + 2) x (bh + 2) pixels with bw = 8, so every image row of the tile is
// one 8-row group of the K-major operand and the group stride (SBO) is bw + 2 rows.  Tap (r, s) reads the same box
// starting r image rows and s pixels further in: a start address that is a whole number of 128-byte rows off the
// swizzle atom, which works because the swizzle is keyed on absolute shared-memory address bits (measured: exact
// results for arbitrary row offsets and group strides).  B tiles come from the resident bank, order [s][cb][r].
template <int KS, bool PAIR>
__device__ __forceinline__ void issue_stage_fh(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t a_hi, uint32_t b_hi, uint32_t idesc,
                                               uint32_t a_row16, uint32_t a_rowpitch16, uint32_t b_tile16, uint32_t b_s16,
                                               uint32_t accumulate_first)
{
#pragma unroll
    for (int sft = 0; sft < 3; ++sft) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                const uint64_t ad = ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + (uint32_t)r * a_rowpitch16 + (uint32_t)sft * a_row16 + 2u * k);
                const uint64_t bd = ((uint64_t)b_hi << 32) | (uint64_t)(b_lo + (uint32_t)sft * b_s16 + (uint32_t)r * b_tile16 + 2u * k);
                const uint32_t acc = (sft == 0 && r == 0 && k == 0) ? accumulate_first : 1u;
                if constexpr (PAIR) umma_bf16_pair(d_tmem, ad, bd, idesc, acc);
                else umma_bf16(d_tmem, ad, bd, idesc, acc);
            }
        }
    }
}

// One MMA-issuing thread.  The CTA runs kIssuers of them (in different warps): issuer `my` accumulates the CTA's units
// my, my + kIssuers, ... (unit j always into accumulator j % acc_bufs) and steps over the ring stages of the others.  A single
// thread cannot keep the tensor pipe busy on narrow tiles: it pays roughly 45 cycles per tcgen05.mma, 180 per barrier
// wait and 55 per commit, all serial, against 48-64 cycles the pipe needs per MMA at N <= 128; two threads working on
// different accumulators can.
template <int KS, int NB, bool PAIR, bool GROUP, bool FH>
__device__ __forceinline__ void mma_issuer(const ConvKParams& p, const UnitWalk& walk, int my, uint32_t tmem_base, uint32_t smem_addr,
                                           uint32_t ring_addr, int stage_bytes, uint64_t* full_bar, uint64_t* empty_bar, uint64_t* acc_full,
                                           uint64_t* acc_empty, uint64_t* w_bar, uint64_t* init_bar, uint32_t* abort_flag, const int* slot_stage)
{
    const uint32_t idesc = make_idesc_bf16(PAIR ? 256 : 128, p.mma_n, false, false);
    const uint32_t sbo = 8u * (uint32_t)p.kb * 2u;  // eight rows of kb bf16
    const uint64_t desc_proto = make_smem_desc(0u, 16u, sbo, (uint32_t)p.swz);
    const uint32_t desc_hi = (uint32_t)(desc_proto >> 32), desc_lo_base = (uint32_t)desc_proto;
    // full halo: A groups are (bw + 2) rows apart
    const uint32_t a_hi_fh = (uint32_t)(make_smem_desc(0u, 16u, (uint32_t)(p.bw + 2) * (uint32_t)p.kb * 2u, (uint32_t)p.swz) >> 32);
    const uint32_t a_row16 = ((uint32_t)p.kb * 2u) >> 4, a_rowpitch16 = (uint32_t)(p.bw + 2) * a_row16;
    const uint32_t b_s16 = (uint32_t)(p.c_blocks * 3 * p.b_bytes) >> 4;
    const uint32_t a_to_b16 = (uint32_t)p.a_bytes >> 4, a_step16 = (uint32_t)p.a_step >> 4;
    // B tiles of consecutive vertical taps are adjacent, in a stage and in the resident bank alike
    const uint32_t b_step16 = (uint32_t)p.b_bytes >> 4;
    const uint32_t b_cb16 = (uint32_t)(p.nb * p.b_bytes) >> 4, stage16 = (uint32_t)stage_bytes >> 4;
    const int G = GROUP ? p.gsub : 1;
    const uint32_t sub16 = GROUP ? stage16 / (uint32_t)G : stage16;   // one k-block inside a slot
    const uint32_t ring_lo = desc_lo_base + (ring_addr >> 4), bank_lo = desc_lo_base + (smem_addr >> 4);
    const int S = p.stages;
    const bool timed = p.stall != nullptr;
    const int units_per_par = p.n_par > 1 ? p.total_units / p.n_par : 1;
    const int n_it_fixed = unit_iters(p, 0);
    bool ok = true;
    if (p.resident && !mbar_wait_warp(w_bar, 0u, p.spin_limit, abort_flag)) {
        atomicOr(p.status, B2C_DEV_TIMEOUT);
        ok = false;
    }
    int s = 0, j = 0, i_stage = 0;   // ring slot and index of the next stage in CTA order, count of units that have stages
    uint32_t ph = 0;
    long long wait_ring = 0, wait_acc = 0;
    for (int pu = walk.first; ok && pu < walk.count; pu += walk.stride) {
        int n_sub = n_it_fixed;   // k-blocks of the unit
        if (p.n_par > 1) n_sub = unit_iters(p, walk.unit(p, pu) / units_per_par);
        if (n_sub == 0) continue;   // a parity without taps: the epilogue stores zeros without an accumulator
        const int n_it = GROUP ? (n_sub + G - 1) / G : n_sub;   // ring slots of the unit
        if ((j % p.issuers) != my) {   // another issuer's unit: step over its stages
            i_stage += n_it;
            s += n_it;
            while (s >= S) { s -= S; ph ^= 1u; }
            ++j;
            continue;
        }
        const int buf = j & (p.acc_bufs - 1);
        const uint32_t d_tmem = tmem_base + (uint32_t)(buf * p.acc_cols);
        uint32_t b_res = bank_lo;   // resident bank: B tile of (tap or horizontal shift, channel block), consecutive per stage
        for (int it = 0; it < n_it; ++it) {
            int n_k = 1;   // k-blocks in this slot
            if constexpr (GROUP) n_k = n_sub - it * G < G ? n_sub - it * G : G;
            const long long w2 = timed ? clock64() : 0;
            // A parity wait tells a barrier's phases apart only modulo two, and with two issuers this thread may reach a
            // slot before the slot's previous stage (another issuer's) was even loaded.  A producer issues the load of
            // stage i only after the previous stage in that slot was consumed, and then stamps the slot with i + 1:
            // seeing the stamp pass i makes the parity wait unambiguous.
            if (p.issuers > 1) {
                uint32_t polls = 0;
                while (__any_sync(0xffffffffu, ld_volatile_shared(&slot_stage[s]) <= i_stage)) {
                    if (++polls > p.spin_limit || __any_sync(0xffffffffu, *(volatile uint32_t*)abort_flag != 0u)) {
                        ok = false;
                        break;
                    }
                }
            }
            if (!ok || !mbar_wait_warp(&full_bar[s], ph, p.spin_limit, abort_flag)) {
                *(volatile uint32_t*)abort_flag = 1u;
                atomicOr(p.status, B2C_DEV_TIMEOUT);
                ok = false;
                break;
            }
            if (timed) wait_ring += clock64() - w2;
            // The accumulator comes second: the unit's first slot is usually full long before the epilogue hands the accumulator
            // back, so the slot's stamp and barrier (600-700 cycles of this thread) are off the path from "accumulator free" to
            // the first MMA, the loop that bounds narrow tiles with two accumulators.
            if (it == 0) {
                const long long w1 = timed ? clock64() : 0;
                if (!mbar_wait_warp(&acc_empty[buf], ((uint32_t)(j >> p.acc_shift) & 1u) ^ 1u, p.spin_limit, abort_flag)) {
                    atomicOr(p.status, B2C_DEV_TIMEOUT);
                    ok = false;
                    break;
                }
                if (timed) wait_acc += clock64() - w1;
            }
            tc_fence_after();
            // descriptors differ from stage to stage only in the 14-bit address field: add offsets to the low word
            if (elect_one()) {
                if constexpr (GROUP) {   // (never with full-halo or merged-tap stages)
                    uint32_t a_lo = ring_lo + (uint32_t)s * stage16;
                    uint32_t b_bank = b_res;
                    for (int g = 0; g < n_k; ++g) {
                        const uint32_t b_lo = p.resident ? b_bank : a_lo + a_to_b16;
                        issue_stage<KS, NB, PAIR>(d_tmem, a_lo, b_lo, desc_hi, idesc, a_step16, b_step16, (it | g) != 0 ? 1u : 0u);
                        b_bank += b_cb16;
                        a_lo += sub16;
                    }
                } else {
                    const uint32_t a_lo = ring_lo + (uint32_t)s * stage16;
                    const uint32_t b_lo = p.resident ? b_res : a_lo + a_to_b16;
                    if constexpr (FH) issue_stage_fh<KS, PAIR>(d_tmem, a_lo, b_lo, a_hi_fh, desc_hi, idesc, a_row16, a_rowpitch16, b_step16, b_s16, it != 0 ? 1u : 0u);
                    else issue_stage<KS, NB, PAIR>(d_tmem, a_lo, b_lo, desc_hi, idesc, a_step16, b_step16, it != 0 ? 1u : 0u);
                }
                // frees the stage (in both CTAs of a pair) once these MMAs have read it
                if constexpr (PAIR) umma_commit_pair(&empty_bar[s], (uint16_t)3);
                else umma_commit(&empty_bar[s]);
            }
            b_res += (uint32_t)n_k * b_cb16;
            __syncwarp();
            ++i_stage;
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (!ok) break;
        if (elect_one()) {
            if constexpr (PAIR) umma_commit_pair(&acc_full[buf], (uint16_t)3);
            else umma_commit(&acc_full[buf]);
        }
        __syncwarp();
        ++j;
    }
    if (timed && elect_one()) {
        atomicAdd(p.stall + 1, (unsigned long long)wait_ring);
        atomicAdd(p.stall + 2, (unsigned long long)wait_acc);
    }
}

// The two MMA-issuing threads of a CTA sharing every unit (tiles wider than 128 channels, where TMEM holds two accumulators
// and the threads cannot take alternate units).  Stage i of the CTA belongs to thread i % 2; the ring depth is even, so
// thread `my` owns the slots my, my + 2, ... and walks them in order with its own phase bit: a slot has one consumer and
// needs no stamp.  Both threads accumulate into the unit's accumulator (accumulation commutes; the tensor pipe runs MMAs
// one after the other).  The thread that does not own a unit's first stage, whose first MMA overwrites the accumulator,
// waits for that stage's completion barrier instead of the accumulator-free barrier (the first stage was issued after
// the accumulator had been freed); both threads commit to the accumulator-full barrier (count 2).  This thread's chain
// of dependent instructions per slot is what bounds these layers, so the loop carries nothing it does not need.
template <int KS, int NB, bool PAIR, bool GROUP>
__device__ __forceinline__ void mma_issuer_split(const ConvKParams& p, const UnitWalk& walk, int my, uint32_t tmem_base, uint32_t smem_addr,
                                                 uint32_t ring_addr, int stage_bytes, uint64_t* full_bar, uint64_t* empty_bar, uint64_t* acc_full,
                                                 uint64_t* acc_empty, uint64_t* w_bar, uint64_t* init_bar, uint32_t* abort_flag)
{
    const uint32_t idesc = make_idesc_bf16(PAIR ? 256 : 128, p.mma_n, false, false);
    const uint64_t desc_proto = make_smem_desc(0u, 16u, 8u * (uint32_t)p.kb * 2u, (uint32_t)p.swz);
    const uint32_t desc_hi = (uint32_t)(desc_proto >> 32), desc_lo_base = (uint32_t)desc_proto;
    const uint32_t a_to_b16 = (uint32_t)p.a_bytes >> 4, a_step16 = (uint32_t)p.a_step >> 4, b_step16 = (uint32_t)p.b_bytes >> 4;
    const uint32_t b_cb16 = (uint32_t)(p.nb * p.b_bytes) >> 4, stage16 = (uint32_t)stage_bytes >> 4;
    const int G = GROUP ? p.gsub : 1;
    const uint32_t sub16 = GROUP ? stage16 / (uint32_t)G : stage16;
    const uint32_t ring_lo = desc_lo_base + (ring_addr >> 4), bank_lo = desc_lo_base + (smem_addr >> 4);
    const int S = p.stages;
    const bool timed = p.stall != nullptr, resident = p.resident != 0;
    const int n_sub_fixed = unit_iters(p, 0);
    const int units_per_par = p.n_par > 1 ? p.total_units / p.n_par : 1;
    long long wait_ring = 0, wait_acc = 0;
    bool ok = true;
    if (resident && !mbar_wait_warp(w_bar, 0u, p.spin_limit, abort_flag)) {
        atomicOr(p.status, B2C_DEV_TIMEOUT);
        ok = false;
    }
    int s = my, k = my;   // this thread's next slot, and the index (in CTA order) of the stage that goes there
    uint32_t ph = 0;
    int i0 = 0, j = 0;    // index of the unit's first stage, count of units with stages
    for (int pu = walk.first; ok && pu < walk.count; pu += walk.stride) {
        int n_sub = n_sub_fixed;
        if (p.n_par > 1) n_sub = unit_iters(p, walk.unit(p, pu) / units_per_par);
        if (n_sub == 0) continue;
        const int i_end = i0 + (GROUP ? (n_sub + G - 1) / G : n_sub);
        const int buf = j & (p.acc_bufs - 1);
        const uint32_t acc_par = (uint32_t)(j >> p.acc_shift) & 1u;
        if (k < i_end) {
            const long long w1 = timed ? clock64() : 0;
            const bool mine_first = k == i0;
            if (!mbar_wait_warp(mine_first ? &acc_empty[buf] : &init_bar[buf], mine_first ? acc_par ^ 1u : acc_par, p.spin_limit, abort_flag)) {
                atomicOr(p.status, B2C_DEV_TIMEOUT);
                ok = false;
                break;
            }
            if (timed) wait_acc += clock64() - w1;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * p.acc_cols);
            do {
                const int it = k - i0;
                const long long w2 = timed ? clock64() : 0;
                if (!mbar_wait_warp(&full_bar[s], ph, p.spin_limit, abort_flag)) {
                    atomicOr(p.status, B2C_DEV_TIMEOUT);
                    ok = false;
                    break;
                }
                if (timed) wait_ring += clock64() - w2;
                tc_fence_after();
                if (elect_one()) {
                    uint32_t a_lo = ring_lo + (uint32_t)s * stage16;
                    if constexpr (GROUP) {
                        const int n_k = n_sub - it * G < G ? n_sub - it * G : G;
                        uint32_t b_res = bank_lo + (uint32_t)(it * G) * b_cb16;
                        for (int g = 0; g < n_k; ++g) {
                            issue_stage<KS, NB, PAIR>(d_tmem, a_lo, resident ? b_res : a_lo + a_to_b16, desc_hi, idesc, a_step16, b_step16, (it | g) != 0 ? 1u : 0u);
                            b_res += b_cb16;
                            a_lo += sub16;
                        }
                    } else {
                        issue_stage<KS, NB, PAIR>(d_tmem, a_lo, resident ? bank_lo + (uint32_t)it * b_cb16 : a_lo + a_to_b16, desc_hi, idesc, a_step16, b_step16,
                                                  it != 0 ? 1u : 0u);
                    }
                    if constexpr (PAIR) umma_commit_pair(&empty_bar[s], (uint16_t)3);   // frees the stage in both CTAs of a pair
                    else umma_commit(&empty_bar[s]);
                    if (it == 0) {   // the overwriting stage (both issuing threads live in the leader CTA of a pair)
                        if constexpr (PAIR) umma_commit_pair(&init_bar[buf], (uint16_t)1);
                        else umma_commit(&init_bar[buf]);
                    }
                }
                __syncwarp();
                k += 2;
                s += 2;
                if (s >= S) { s = my; ph ^= 1u; }
            } while (k < i_end);
            if (!ok) break;
        } else if (!mbar_wait_warp(&acc_empty[buf], acc_par ^ 1u, p.spin_limit, abort_flag)) {
            // No stage of this unit is this thread's (units of one slot).  Its commit still counts towards the accumulator's barrier, so it
            // must not run ahead of the buffer's previous unit: two commits of this thread would complete that unit's phase early.
            atomicOr(p.status, B2C_DEV_TIMEOUT);
            ok = false;
            break;
        }
        if (elect_one()) {
            if constexpr (PAIR) umma_commit_pair(&acc_full[buf], (uint16_t)3);
            else umma_commit(&acc_full[buf]);
        }
        __syncwarp();
        i0 = i_end;
        ++j;
    }
    if (timed && elect_one()) {
        atomicAdd(p.stall + 1, (unsigned long long)wait_ring);
        atomicAdd(p.stall + 2, (unsigned long long)wait_acc);
    }
}

// The kernel comes in four kinds, one per family of launch plans, so that each carries only the issuing and epilogue code its
// plans use (with all of them in one kernel the code of a launch was spread over several hundred KB and the 64- and
// 128-channel layers ran 7-12 % slower inside a training step, where every launch starts on a cold instruction cache):
// general (one MMA per tap or vertical tap reuse, any tile width up to 128 channels), split (tiles wider than 128 channels:
// two issuing threads share every unit), merged horizontal taps, full-halo stages.
enum : int { KIND_GENERAL = 0, KIND_SPLIT = 1, KIND_HMERGE = 2, KIND_FULL_HALO = 3 };
// BLOCKS: with epilogue_blocks in place of epilogue_loop (p.block_cols).
template <bool PAIR, int KIND, bool BLOCKS>
__global__ void __launch_bounds__(kThreads, 1) conv_kmajor_kernel(const __grid_constant__ ConvKParams p)
{
    const int rank = PAIR ? (int)cluster_ctarank() : 0;   // 0 = leader of the pair: issues the MMAs, owns the barriers the pair shares
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_full[kMaxAccBufs], acc_empty[kMaxAccBufs], init_bar[kMaxAccBufs], w_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ uint32_t abort_flag;
    __shared__ int slot_stage[kMaxStages];   // per ring slot: 1 + index of the stage whose loads were issued into it last
    __shared__ int2 s_last;   // statistics group and channel tile whose sums the epilogue warps left in s_stats
    __shared__ __align__(16) float s_stats[kEpiWarps][256];   // per epilogue warp (128 columns at most): [0,128) sums, [128,256) sums of squares

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~uintptr_t(1023));
    uint8_t* ring = smem + p.resident_bytes;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // the compiler sees a warp-uniform role
    const int S = p.stages;
    const int sub_bytes = p.a_bytes + (p.resident ? 0 : p.nb * p.b_bytes);   // one k-block: the A tile and, unless the bank is resident, its filter tiles
    const int stage_bytes = p.gsub * sub_bytes;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < kMaxAccBufs; ++b) {
            mbar_init(&acc_full[b], p.issue_split ? 2 : 1);   // shared units: both issuing threads commit
            mbar_init(&init_bar[b], 1);
            mbar_init(&acc_empty[b], PAIR ? 2 * kEpiWarps : kEpiWarps);   // one arrival per epilogue warp (of both CTAs of a pair)
        }
        mbar_init(&w_bar, 1);
        mbar_init(&drain_bar, kIssuers);
        abort_flag = 0;
        for (int i = 0; i < kMaxStages; ++i) slot_stage[i] = 0;
        fence_mbar_init();
    }
    const UnitWalk walk(p, rank);   // (its divisions are over before the wait for the previous kernel)
    if (warp == 1) {
        if constexpr (PAIR) {
            tmem_alloc_pair(&tmem_slot, (uint32_t)p.tmem_cols);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(&tmem_slot, (uint32_t)p.tmem_cols);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();   // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    // set-up done (it touched no global data): order behind the previous kernel of the stream, then let the next one in
    pdl_begin(p.no_wait);
    const long long t_start = clock64();
    int last_issued = -1;  // producer lanes: index of the last stage whose loads this lane issued

    if (warp == 0 || warp == kProducerWarp1) {
        {
            // ------------------------------------------------------------ TMA producers
            // Producer w fills the ring slots w, w + kProducers, ...: the chain wait -> expect -> issue of one thread
            // (several hundred cycles) would otherwise bound short stages.  Splitting by slot (not by stage) keeps
            // every slot with one producer that uses it strictly in order, which a parity wait on its barrier needs.
            const int w = warp == 0 ? 0 : 1;
            if (elect_one()) {
                prefetch_tensormap(&p.tmB);
                prefetch_tensormap(&p.tmA[0]);
            }
            // a pair counts the bytes of both CTAs on the leader's barriers; b_row = first filter row this CTA fetches
            const int b_rows = PAIR ? p.n_tile >> 1 : p.n_tile;
            const int R = p.r_filter;
            const uint32_t w_bar_cl = PAIR ? map_to_cta(smem_u32(&w_bar), 0) : 0u;
            if (KIND == KIND_HMERGE && w == 0 && elect_one()) {
                // merged horizontal taps: per channel block one box of all nine taps, landing as [r][s][out][64 in]:
                // three tiles (one per filter row) of 3 x n_tile rows
                const int oc0 = (walk.first % p.n_ktiles) * p.n_tile;
                mbar_expect_tx(&w_bar, (uint32_t)(p.c_blocks * 3 * p.tx_b));
                for (int cb = 0; cb < p.c_blocks; ++cb)
                    tma_load_4d(smem + (size_t)cb * 3 * p.b_bytes, &p.tmB, &w_bar, cb * p.kb, oc0, 0, 0);
            } else if (KIND != KIND_HMERGE && p.resident && w == 0 && elect_one()) {
                // bank order: [tap or horizontal shift][channel block][vertical tap]
                const int ktile = walk.first % p.n_ktiles;   // the walk stride is a multiple of n_ktiles: fixed per CTA
                const TapList& tl = p.taps[0];
                const int oc0 = ktile * p.n_tile + rank * b_rows;
                if (rank == 0) mbar_expect_tx(&w_bar, (uint32_t)((PAIR ? 2 : 1) * tl.count * p.c_blocks * p.tx_b));
                const int groups = (p.vreuse || p.fh) ? tl.count / 3 : tl.count;
                for (int t = 0; t < groups; ++t)
                    for (int cb = 0; cb < p.c_blocks; ++cb) {
                        uint8_t* dst = smem + (size_t)(t * p.c_blocks + cb) * p.nb * p.b_bytes;
                        const int n_loads = p.b_merged ? 1 : p.nb;
                        for (int v = 0; v < n_loads; ++v) {
                            const int rs = tl.rs[t + 3 * v];
                            if constexpr (PAIR) tma_load_4d_pair(dst + (size_t)v * p.b_bytes, &p.tmB, w_bar_cl, cb * p.kb, rs % R, oc0, rs / R);
                            else tma_load_4d(dst + (size_t)v * p.b_bytes, &p.tmB, &w_bar, cb * p.kb, rs % R, oc0, rs / R);
                        }
                    }
            }
            __syncwarp();
            bool ok = true;
            long long waited = 0;
            const bool timed = p.stall != nullptr;
            int i = w, i_base = 0;   // this producer's next stage and the first stage of the current unit, in CTA order
            int s = w;   // w < kProducers <= S
            uint32_t ph = 0u;
            const uint32_t stage_tx = (uint32_t)(p.tx_a + (p.resident ? 0 : p.nb * p.tx_b));
            const int n_b_loads = p.resident ? 0 : (p.b_merged ? 1 : p.nb);
            for (int pu = walk.first; ok && pu < walk.count; pu += walk.stride) {
                const int u = walk.unit(p, pu);
                const int n_sub = unit_iters(p, p.n_par > 1 ? u / (p.total_units / p.n_par) : 0);
                const int G = (KIND == KIND_GENERAL || KIND == KIND_SPLIT) ? p.gsub : 1;   // (full-halo and merged-tap stages are never grouped)
                const int n_it = G > 1 ? (n_sub + G - 1) / G : n_sub;   // ring slots of the unit
                if (i >= i_base + n_it) {   // no stage of this unit is mine
                    i_base += n_it;
                    continue;
                }
                const UnitCoord c = decode_unit(p, u);
                const TapList& tl = p.taps[c.par];
                const int oc0 = c.ktile * p.n_tile + rank * b_rows;
                while (i < i_base + n_it) {
                    const int it = i - i_base;
                    // waits until the slot's previous stage has been consumed; that stage's barrier phase is then over, and the
                    // stamp lets issuers that take alternate units tell the slot's phases apart (a relaxed store: the wait orders it)
                    auto wait_empty = [&]() -> bool {
                        const long long w0 = timed ? clock64() : 0;
                        if (!mbar_wait_warp(&empty_bar[s], ph ^ 1u, p.spin_limit, &abort_flag)) {
                            atomicOr(p.status, B2C_DEV_TIMEOUT);
                            ok = false;
                            return false;
                        }
                        if (timed) waited += clock64() - w0;
                        if (p.issuers > 1 && !p.issue_split && lane == 0) st_volatile_shared(&slot_stage[s], i + 1);
                        return true;
                    };
                    if (G > 1) {
                        if (!wait_empty()) break;
                        // the k-blocks that share this slot (one, except where short k-blocks are grouped)
                        const int k_first = it * G, n_k = n_sub - k_first < G ? n_sub - k_first : G;
                        if (elect_one()) {
                            if constexpr (PAIR) {
                                if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * (uint32_t)n_k * stage_tx);
                            } else {
                                mbar_expect_tx(&full_bar[s], (uint32_t)n_k * stage_tx);
                            }
                            for (int g = 0; g < n_k; ++g) {
                                const int kblk = k_first + g;
                                const int t0 = p.cb_shift >= 0 ? kblk >> p.cb_shift : kblk / p.c_blocks;   // tap
                                const int cb = kblk - t0 * p.c_blocks;                                       // channel block
                                uint8_t* a_dst = ring + (size_t)s * stage_bytes + (size_t)g * sub_bytes;
                                if constexpr (PAIR) {
                                    const uint32_t full_cl = map_to_cta(smem_u32(&full_bar[s]), 0);
                                    tma_load_4d_pair(a_dst, &p.tmA[tl.map[t0]], full_cl, cb * p.kb, c.ow0 + tl.dw[t0], c.oh0 + tl.dh[t0], c.n0);
                                    for (int v = 0; v < n_b_loads; ++v) {
                                        const int rs = tl.rs[t0 + 3 * v], fr = (rs * 11) >> 5;   // rs / 3 for rs < 9 (R is 1 or 3)
                                        tma_load_4d_pair(a_dst + p.a_bytes + (size_t)v * p.b_bytes, &p.tmB, full_cl, cb * p.kb, rs - fr * R, oc0, fr);
                                    }
                                } else {
                                    tma_load_4d(a_dst, &p.tmA[tl.map[t0]], &full_bar[s], cb * p.kb, c.ow0 + tl.dw[t0], c.oh0 + tl.dh[t0], c.n0);
                                    for (int v = 0; v < n_b_loads; ++v) {
                                        const int rs = tl.rs[t0 + 3 * v], fr = (rs * 11) >> 5;   // rs / 3 for rs < 9 (R is 1 or 3)
                                        tma_load_4d(a_dst + p.a_bytes + (size_t)v * p.b_bytes, &p.tmB, &full_bar[s], cb * p.kb, rs - fr * R, oc0, fr);
                                    }
                                }
                            }
                        }
                    } else {
                        // (operands first, the wait second: the address arithmetic is off the chain wait -> expect -> issue)
                        int t0 = p.cb_shift >= 0 ? it >> p.cb_shift : it / p.c_blocks;   // tap (or horizontal shift)
                        const int cb = it - t0 * p.c_blocks;                               // channel block
                        if (KIND == KIND_HMERGE || KIND == KIND_FULL_HALO) t0 = 0;   // one box per channel block: the entry of tap (0, 0) carries its origin
                        uint8_t* a_dst = ring + (size_t)s * stage_bytes;
                        // with vreuse the table entry of vertical tap 0 carries the shift of the whole haloed tile
                        const CUtensorMap* map_a = &p.tmA[tl.map[t0]];
                        const int ca = cb * p.kb, wa = c.ow0 + (KIND == KIND_HMERGE ? 0 : tl.dw[t0]), ha = c.oh0 + tl.dh[t0];   // merged taps: no horizontal shift
                        int b_s[3], b_r[3];
#pragma unroll
                        for (int v = 0; v < 3; ++v) {
                            const int rs = v < n_b_loads ? tl.rs[t0 + 3 * v] : 0, fr = (rs * 11) >> 5;   // rs / 3 for rs < 9 (R is 1 or 3)
                            b_s[v] = rs - fr * R;
                            b_r[v] = fr;
                        }
                        if (!wait_empty()) break;
                        if (elect_one()) {
                            if constexpr (PAIR) {
                                const uint32_t full_cl = map_to_cta(smem_u32(&full_bar[s]), 0);
                                if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * stage_tx);
                                tma_load_4d_pair(a_dst, map_a, full_cl, ca, wa, ha, c.n0);
#pragma unroll
                                for (int v = 0; v < 3; ++v)
                                    if (v < n_b_loads) tma_load_4d_pair(a_dst + p.a_bytes + (size_t)v * p.b_bytes, &p.tmB, full_cl, ca, b_s[v], oc0, b_r[v]);
                            } else {
                                mbar_expect_tx(&full_bar[s], stage_tx);
                                tma_load_4d(a_dst, map_a, &full_bar[s], ca, wa, ha, c.n0);
#pragma unroll
                                for (int v = 0; v < 3; ++v)
                                    if (v < n_b_loads) tma_load_4d(a_dst + p.a_bytes + (size_t)v * p.b_bytes, &p.tmB, &full_bar[s], ca, b_s[v], oc0, b_r[v]);
                            }
                        }
                    }
                    __syncwarp();
                    last_issued = i;
                    if (s + kProducers < S) {
                        i += kProducers;
                        s += kProducers;
                    } else {   // wrap to this producer's first slot
                        i += S - s + w;
                        s = w;
                        ph ^= 1u;
                    }
                }
                i_base += n_it;
            }
            if (p.stall != nullptr && rank == 0 && w == 0 && lane == 0) {
                atomicAdd(p.stall + 0, (unsigned long long)waited);
                atomicAdd(p.stall + 4, (unsigned long long)(clock64() - t_start));
            }
        }
    } else if (warp == 1 || (warp >= 2 + kEpiWarps && warp < kProducerWarp1)) {
        if (rank == 0) {
            // ------------------------------------------------------------ MMA issuers (in the leader CTA of a pair)
            const int my = warp == 1 ? 0 : warp - (2 + kEpiWarps) + 1;
            if (my < p.issuers) {
                const uint32_t smem_addr = smem_u32(smem), ring_addr = smem_u32(ring);
                const int ksteps = p.kb >> 4;
                if constexpr (KIND == KIND_SPLIT) {
#define B2C_ISSUER_S(KS, NB, GR) mma_issuer_split<KS, NB, PAIR, GR>(p, walk, my, tmem_base, smem_addr, ring_addr, stage_bytes, full_bar, empty_bar, acc_full, acc_empty, &w_bar, init_bar, &abort_flag)
                    if (p.nb == 3) {
                        if (ksteps == 4) B2C_ISSUER_S(4, 3, false);
                        else if (ksteps == 2) B2C_ISSUER_S(2, 3, false);
                        else B2C_ISSUER_S(1, 3, false);
                    } else if (p.gsub > 1) {
                        if (ksteps == 4) B2C_ISSUER_S(4, 1, true);
                        else if (ksteps == 2) B2C_ISSUER_S(2, 1, true);
                        else B2C_ISSUER_S(1, 1, true);
                    } else {
                        if (ksteps == 4) B2C_ISSUER_S(4, 1, false);
                        else if (ksteps == 2) B2C_ISSUER_S(2, 1, false);
                        else B2C_ISSUER_S(1, 1, false);
                    }
#undef B2C_ISSUER_S
                } else {
#define B2C_ISSUER(KS, NB, GR, FH) mma_issuer<KS, NB, PAIR, GR, FH>(p, walk, my, tmem_base, smem_addr, ring_addr, stage_bytes, full_bar, empty_bar, acc_full, acc_empty, &w_bar, init_bar, &abort_flag, slot_stage)
                    if constexpr (KIND == KIND_HMERGE) {
                        B2C_ISSUER(4, 3, false, false);   // 64-channel k-blocks, the three filter rows of a channel block per stage
                    } else if constexpr (KIND == KIND_FULL_HALO) {
                        B2C_ISSUER(4, 3, false, true);
                    } else if (p.nb == 3) {
                        if (ksteps == 4) B2C_ISSUER(4, 3, false, false);
                        else if (ksteps == 2) B2C_ISSUER(2, 3, false, false);
                        else B2C_ISSUER(1, 3, false, false);
                    } else if (p.gsub > 1) {
                        if (ksteps == 4) B2C_ISSUER(4, 1, true, false);
                        else if (ksteps == 2) B2C_ISSUER(2, 1, true, false);
                        else B2C_ISSUER(1, 1, true, false);
                    } else {
                        if (ksteps == 4) B2C_ISSUER(4, 1, false, false);
                        else if (ksteps == 2) B2C_ISSUER(2, 1, false, false);
                        else B2C_ISSUER(1, 1, false, false);
                    }
#undef B2C_ISSUER
                }
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue (8 warps)
        const int e = warp - 2;
        int2 last;
#define B2C_EPILOGUE(NCH, EAGER, HM)                                                                                                           \
    last = p.stats != nullptr ? epilogue_loop<NCH, EAGER, HM, true>(p, tmem_base, acc_full, acc_empty, &abort_flag, s_stats[e], e, lane, rank) \
                              : epilogue_loop<NCH, EAGER, HM, false>(p, tmem_base, acc_full, acc_empty, &abort_flag, s_stats[e], e, lane, rank)
#define B2C_BLOCKS(BC, NB, HM)                                                                                                                            \
    last = p.stats != nullptr ? epilogue_blocks<BC, NB, HM, true>(p, tmem_base, acc_full, acc_empty, &abort_flag, s_stats[e], stage, e, lane, rank) \
                              : epilogue_blocks<BC, NB, HM, false>(p, tmem_base, acc_full, acc_empty, &abort_flag, s_stats[e], stage, e, lane, rank)
        if constexpr (BLOCKS) {
            // (s_stats, which is written once all epilogue warps are through with their blocks, has room for two blocks of 64 columns, or for the
            // eight of 16)
            uint8_t* spare = reinterpret_cast<uint8_t*>(s_stats);
            uint8_t* behind = ring + (size_t)S * stage_bytes;
            uint8_t* stage = p.block_cols == 16 ? spare + 1024 * e : p.block_cols == 32 ? behind + 2048 * e : e < 2 ? spare + 4096 * e : behind + 4096 * (e - 2);
            if constexpr (KIND == KIND_SPLIT) B2C_BLOCKS(64, 2, false);
            else if constexpr (KIND == KIND_HMERGE) B2C_BLOCKS(32, 1, true);
            else if constexpr (KIND == KIND_FULL_HALO) B2C_BLOCKS(16, 4, false);
            else if (p.n_tile == 64) B2C_BLOCKS(32, 1, false);
            else B2C_BLOCKS(64, 1, false);
        } else if constexpr (KIND == KIND_SPLIT) {   // tiles wider than 128 channels
            B2C_EPILOGUE(8, false, false);
        } else if constexpr (KIND == KIND_HMERGE) {
            B2C_EPILOGUE(2, true, true);
        } else {
            if (KIND == KIND_GENERAL && p.n_tile <= 32 && !p.out_is_f32) B2C_EPILOGUE(1, true, false);
            else if (p.n_tile <= 64 && !p.out_is_f32) B2C_EPILOGUE(2, true, false);
            else if (KIND == KIND_FULL_HALO || p.n_tile <= 128) B2C_EPILOGUE(4, false, false);
            else B2C_EPILOGUE(8, false, false);   // (only with issue splitting switched off)
        }
#undef B2C_EPILOGUE
#undef B2C_BLOCKS
        if (e == 0 && lane == 0) s_last = last;
    }
    tc_fence_before();
    __syncthreads();
    if (p.stats != nullptr && !abort_flag && s_last.x >= 0) {   // the last statistics group of this CTA
        const int first_half = (((p.n_tile >> 4) + 1) >> 1) * 16;
        double* st = p.stats + (size_t)s_last.x * 2 * p.oc_valid + s_last.y * p.n_tile;
        for (int i = threadIdx.x; i < p.n_tile; i += kThreads) {
            const int half = i >= first_half ? 1 : 0, col = i - half * first_half;
            double s = 0.0, sq = 0.0;
            for (int q = 0; q < 4; ++q) {
                s += (double)s_stats[half * 4 + q][col];
                sq += (double)s_stats[half * 4 + q][128 + col];
            }
            atomicAdd(st + i, s);
            atomicAdd(st + p.oc_valid + i, sq);
        }
        __syncwarp();
    }
    if constexpr (PAIR) cluster_sync_all();   // both CTAs have left their loops: nothing new will be issued
    if (abort_flag) {
        // A wait gave up.  Before the CTA may exit, let every bulk copy it issued land and every
        // MMA it issued retire (both finish on their own; the polls here only bound the wait).
        // In a pair the leader's barriers count the peer's copies too.
        if ((warp == 0 || warp == kProducerWarp1) && lane == 0 && rank == 0) {
            if (p.resident && warp == 0)
                for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(&w_bar, 0u); ++i) {}
            // the last stage issued into each of the own slots (older ones were consumed, so they had landed)
            const int w = warp == 0 ? 0 : 1;
            for (int sl = w; sl < S; sl += kProducers) {
                if (last_issued < sl) continue;
                const int it = last_issued - ((last_issued - sl) % S);   // largest stage index <= last_issued in slot sl
                for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(&full_bar[sl], (uint32_t)(it / S) & 1u); ++i) {}
            }
        }
        if ((warp == 1 || (warp >= 2 + kEpiWarps && warp < kProducerWarp1)) && rank == 0 && elect_one()) {   // a commit covers the MMAs of the thread that makes it
            if constexpr (PAIR) umma_commit_pair(&drain_bar, (uint16_t)1);
            else umma_commit(&drain_bar);
            if (warp == 1)
                for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(&drain_bar, 0u); ++i) {}
        }
        __syncthreads();
    }
    if constexpr (PAIR) cluster_sync_all();   // the peer must not exit while the leader still drains copies into it
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, (uint32_t)p.tmem_cols);
        else tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
    pdl_end(p.no_wait);
}

// ------------------------------------------------------------------------------------------ host side
static bool encode_map(b2c_ctx* ctx, CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
                       const cuuint32_t* box, int inner_bytes)
{
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUtensorMapSwizzle swz = inner_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : inner_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    CUresult r = ctx->encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides_bytes, box, estr,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Activation tensor [n][h][w][c] viewed with a spatial step (1: plain; 2: one parity of rows/cols).
bool encode_activation_map(b2c_ctx* ctx, CUtensorMap* tm, const void* base, int n, int h, int w, int c, int step, int ph, int pw, int box_c,
                           int box_w, int box_h, int box_n)
{
    const char* b = reinterpret_cast<const char*>(base) + ((size_t)ph * w + pw) * c * 2;
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)(w / step), (cuuint64_t)(h / step), (cuuint64_t)n};
    cuuint64_t str[3] = {(cuuint64_t)step * c * 2, (cuuint64_t)step * w * c * 2, (cuuint64_t)h * w * c * 2};
    cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)box_n};
    return encode_map(ctx, tm, b, 4, dims, str, box, box_c * 2);
}

static int log2_exact(int v)
{
    if (v <= 0 || (v & (v - 1)) != 0) return -1;
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

static int floordiv2(int e) { return (e >= 0) ? e / 2 : -((-e + 1) / 2); }

void forward_taps(TapList& tl, int R, int stride, int pad)
{
    tl.count = 0;
    for (int r = 0; r < R; ++r)
        for (int s = 0; s < R; ++s) {
            const int i = tl.count++;
            const int eh = r - pad, ew = s - pad;
            if (stride == 1) {
                tl.map[i] = 0; tl.dh[i] = (int8_t)eh; tl.dw[i] = (int8_t)ew;
            } else {
                const int hp = eh & 1, wp = ew & 1;
                tl.map[i] = (int8_t)(hp * 2 + wp);
                tl.dh[i] = (int8_t)floordiv2(eh);
                tl.dw[i] = (int8_t)floordiv2(ew);
            }
            tl.rs[i] = (int8_t)(r * R + s);
        }
}

// A launch plan: the kernel's parameter block (tensor maps included), launch shape and shared-memory size.
struct KMajorPlan {
    ConvKParams p;
    int grid;
    size_t smem_bytes;
};

// Tensor-pipe and staging cycles of one k-block of kb channels on a tile of 128 pixels (a pair: 2 x 128) x n channels: an MMA of 16
// channels takes n / 2 cycles, or what its operands take through the 128 B/clk shared-memory port (A: 4 KB, B: 32 n bytes, half of
// it per CTA of a pair); the loads come in at about 74 B/clk per SM, 52 where the tile's width is no power of
// two (fitted with the estimates below, where 160- and 80-channel tiles weigh most).
static int kblock_cycles(int n, int kb, bool pair, int a_rows)
{
    const int b_rows = pair ? n / 2 : n;
    const int operand = 32 + b_rows / 4, mma = (operand > n / 2 ? operand : n / 2) * (kb / 16);
    const int loads = (a_rows + b_rows) * kb * 2 / ((n & (n - 1)) && kb == 64 ? 52 : 74);
    return mma > loads ? mma : loads;
}

// Plan for the one-wave kernel (conv_splitk.cu) for a problem whose tiles do not fill the chip, or false where the persistent
// plan (est_cycles) is the better one.  A cluster of `splits` CTAs or pairs shares a tile's k-blocks and adds the partial tiles
// up at the end; splits = 1 is a tile per CTA or pair, whose shorter epilogue still beats the persistent kernel's one unit.
// The estimates, in cycles over the 4 us that any launch takes, were fitted to timed plans.  K-blocks of 64 channels: 187 layers, the plan
// they pick is on average 5 % slower than the layer's best one (most of that on short reductions, which stay whole).  Narrower ones, whose
// rows of 32 and 64 bytes come in more slowly, have constants of their own: 503 layers, on average 1.1 % and at most 28 % slower than
// the best plan, where those of the wide ones picked plans up to 2.7 times as slow (25 images, 784 -> 512 at 16x16 55 us in the persistent
// kernel, 97 in the plan that they preferred; 17 images, 160 -> 160 at 32x32 12.0 and 15.6).  With 128 images, persistent -> this, launch to
// launch: 512 -> 512 at 4x4 27.8 -> 13.6 us, 256 -> 256 at 8x8 18.2 -> 12.3, 256 -> 512 at 8x8 stride 2 16.6 -> 10.3; with 50
// images 26.3 -> 10.4, 16.4 -> 9.8 and 16.4 -> 8.2; 128 -> 128 at 8x8 with 16 images 10.3 -> 6.3.
static bool choose_splitk(b2c_ctx* ctx, const KMajorProblem& pb, ConvKParams& p, int m_tiles, bool reuse, long long est_cycles)
{
    const int kb = (pb.ic % 64 == 0) ? 64 : (pb.ic % 32 == 0) ? 32 : 16;
    const int taps = p.n_par > 1 ? ((pb.r + 1) / 2) * ((pb.r + 1) / 2) : pb.r * pb.r;   // of the parity with most
    const int min_taps = p.n_par > 1 ? 1 : taps;
    const int c_blocks = pb.ic / kb;
    const bool narrow = kb < 64;
    // worth a change from the persistent kernel: 0.6 us, and a quarter where that one shares loads and the estimates are less sure
    long long best = (narrow && reuse ? est_cycles * 18 / 25 : est_cycles) - 600;
    bool found = false;
    for (int pair = 0; pair <= 1; ++pair) {
        if (pair && (p.n_par > 1 || ctx->use_pairs == 0)) continue;
        for (int n = 256; n >= 32; n -= 16) {
            if (pb.oc % n || (pair && n % 32)) continue;
            const int clusters = p.n_par * (pair ? (m_tiles / p.n_par + 1) / 2 : m_tiles / p.n_par) * (pb.oc / n);
            for (int splits = 1; splits * (pair + 1) <= 8; splits *= 2) {
                if (n % (8 * splits) || splits > min_taps * c_blocks) continue;
                // (short reductions stay whole: a split saves them a microsecond at most)
                if (splits > 1 && est_cycles < 15000) continue;
                // two tiles per SM: their CTAs (72 registers, half of the shared memory each) take turns at the tensor pipe, one in
                // its epilogue while the other loads.  (The occupancy calculator answers one for kernels that allocate TMEM, so it is
                // not asked; 191 CTAs that live 19.0 k cycles each start every 17 k cycles.)
                const bool two = splits == 1 && !pair && !reuse && clusters > ctx->sm_count && clusters <= 2 * ctx->sm_count;
                if (!two && clusters > splitk_max_clusters(ctx, splits * (pair + 1), pair != 0)) continue;
                const int smem = (two ? 94 : 208) * 1024;   // (beside 16.6 KB of static arrays)
                const int b_rows = pair ? n / 2 : n, a_bytes = 128 * kb * 2, b_bytes = (b_rows * kb * 2 + 1023) & ~1023;
                const int x_bytes = (splits - 1) * (n / splits) * 512;   // partial tiles of the other CTAs
                // k-blocks share a slot until it holds the MMAs of the issuing thread's 500 cycles per slot, while three slots are left
                const int block = kblock_cycles(n, kb, pair != 0, 128), mma = (n / 2 > 48 ? n / 2 : 48) * (kb / 16);
                int gsub = 1;
                while (gsub < 4 && gsub * mma < 480 && 6 * gsub * (a_bytes + b_bytes) <= smem && 2 * gsub * splits <= taps * c_blocks) gsub *= 2;
                const int slot = gsub * (a_bytes + b_bytes);
                int stages = (smem - x_bytes) / slot;
                const int overlap = splits > 1 && stages < (gsub > 1 ? 3 : 4) ? 1 : 0;   // too few slots left: exchange through the ring's memory
                if (overlap) stages = smem / slot;
                if (stages > kMaxStages) stages = kMaxStages;
                if (stages < 2 || (overlap && stages * slot < x_bytes)) continue;
                const int k_blocks = (taps * c_blocks + splits - 1) / splits;
                // k-blocks, exchange (barriers, partial tiles at 21 B/clk), epilogue of n / splits columns.  A slot of narrow k-blocks takes
                // 1900 cycles however little it holds, most of them latency, which two tiles per SM hide for each other.
                const int slot_cycles = narrow ? 1900 : 570, own = narrow && two ? 2 * block : block;
                const long long per_block = own > slot_cycles / gsub ? own : slot_cycles / gsub;
                const long long est = k_blocks * per_block * (two && !narrow ? 2 : 1) + (two ? 2000 : 0) + (splits > 1 ? (narrow ? 1700 : 1100) + 800 * overlap + x_bytes / 21 : 0) +
                                      190ll * n / splits / 32 + (narrow ? 5000 : 2600) * pair;
                if (est >= best) continue;
                best = est;
                found = true;
                p.n_tile = n; p.n_ktiles = pb.oc / n; p.pair = pair; p.splits = splits;
                p.a_bytes = a_bytes; p.b_bytes = b_bytes; p.gsub = gsub; p.stages = stages;
                p.x_overlap = overlap;
                p.x_off = overlap ? 0 : stages * slot;
            }
        }
    }
    if (!found) return false;
    const int b_rows = p.pair ? p.n_tile / 2 : p.n_tile;
    p.kb = kb; p.c_blocks = c_blocks;
    p.swz = kb == 64 ? SWZ_128B : kb == 32 ? SWZ_64B : SWZ_32B;
    p.nb = 1;
    p.tx_a = p.a_bytes;
    p.tx_b = b_rows * kb * 2;
    p.tmem_cols = 32;
    while (p.tmem_cols < p.n_tile) p.tmem_cols *= 2;
    p.total_units = p.n_par * (p.pair ? m_tiles + (m_tiles & 1) : m_tiles / p.n_par) * p.n_ktiles;
    return true;
}

static b2c_status build_kmajor_plan(b2c_ctx* ctx, const KMajorProblem& pb, KMajorPlan& plan)
{
    ConvKParams& p = plan.p;
    memset(&plan, 0, sizeof(plan));
    const int R = pb.r;
    if (!(R == 1 || R == 3) || !(pb.stride == 1 || pb.stride == 2) || pb.pad != (R - 1) / 2) return B2C_ERR_UNSUPPORTED_SHAPE;
    if (pb.n < 1 || pb.ic < 16 || pb.ic % 16 || pb.oc < 16 || pb.oc % 16) return B2C_ERR_UNSUPPORTED_SHAPE;
    // tile grid = spatial grid each unit's 128 accumulator rows walk over
    int gh, gw, n_par = 1;
    if (!pb.dgrad) {
        gh = pb.oh; gw = pb.ow;
        if (pb.ih != pb.oh * pb.stride || pb.iw != pb.ow * pb.stride) return B2C_ERR_UNSUPPORTED_SHAPE;
    } else {
        gh = pb.ih; gw = pb.iw;  // the dy grid; for stride 2 each parity of dx has exactly this size
        if (pb.oh != pb.ih * pb.stride || pb.ow != pb.iw * pb.stride) return B2C_ERR_UNSUPPORTED_SHAPE;
        n_par = pb.stride * pb.stride;
    }
    if (!b2c_is_pow2(gh) || !b2c_is_pow2(gw) || gh > 128 || gw > 128) return B2C_ERR_UNSUPPORTED_SHAPE;
    if (!b2c_aligned16(pb.in) || !b2c_aligned16(pb.wt) || !b2c_aligned16(pb.out)) return B2C_ERR_MISALIGNED;

    p.bw = gw < 128 ? gw : 128;
    p.bh = (128 / p.bw) < gh ? (128 / p.bw) : gh;
    p.bn = 128 / (p.bw * p.bh);
    p.tiles_w = gw / p.bw;
    p.tiles_h = gh / p.bh;
    p.tiles_n = (pb.n + p.bn - 1) / p.bn;
    p.n_par = n_par;

    // output-channel tile: the largest multiple of 16 up to 256 that splits oc evenly
    int n_tile = 16;
    for (int cand = 256; cand >= 16; cand -= 16)
        if (pb.oc % cand == 0) { n_tile = cand; break; }
    p.n_tile = n_tile;
    p.n_ktiles = pb.oc / n_tile;
    p.acc_cols = ((n_tile + 31) / 32) * 32;
    // four accumulators where TMEM has room: the issuers then run a unit or two ahead of the epilogue
    p.acc_bufs = (4 * p.acc_cols <= 512) ? 4 : 2;
    p.acc_shift = p.acc_bufs == 4 ? 2 : 1;
    p.tmem_cols = 32;
    while (p.tmem_cols < p.acc_bufs * p.acc_cols) p.tmem_cols *= 2;
    p.total_units = n_par * p.tiles_n * p.tiles_h * p.tiles_w * p.n_ktiles;

    // CTA pairs (cta_group::2): two neighbouring pixel tiles share every filter tile, each CTA holding half of its
    // rows, which halves the shared-memory operand traffic per MMA.  Needs an even number of pixel tiles and a channel
    // tile that splits into two multiples of 16; the fp32 / bias / multi-parity cases stay on single CTAs.
    const int m_tiles = p.tiles_n * p.tiles_h * p.tiles_w;
    // Measured on B200 (1024-image layers): pairs gain ~30 % at 128-channel tiles, where the filter traffic from L2
    // bounds single CTAs, and lose 5-30 % at 64 channels and on the short reductions of 1x1 and stride-2 layers; so by
    // default only 3x3 stride-1 layers with tiles of 128 channels and more use them (use_pairs: 0 = never, 1 = those, 2 = every
    // eligible problem, 3 = 128-channel tiles only).  Where single CTAs get by with one tile each, short reductions are faster without
    // the pair's set-up and longer operand path: 160 -> 160 at 32x32 with 16 images 15.1 us as pairs, 11.6 as singles, 128 -> 128 at
    // 16x16 with 50 10.4 and 8.3, but 320 -> 320 at 16x16 with 32 16.6 and 17.2.
    const bool pair_ok = n_par == 1 && !pb.out_f32 && pb.bias == nullptr && n_tile % 32 == 0 && m_tiles % 2 == 0 && ctx->sm_count >= 2;
    const bool short_wave = p.total_units <= ctx->sm_count && R * R * pb.ic < 2048;
    p.pair = (pair_ok && (ctx->use_pairs == 2 || (ctx->use_pairs == 1 && n_tile >= 128 && R == 3 && pb.stride == 1 && !short_wave) ||
                          (ctx->use_pairs == 3 && n_tile == 128 && R == 3 && pb.stride == 1))) ? 1 : 0;
    int b_rows = p.pair ? n_tile / 2 : n_tile;   // filter rows one CTA fetches per tile

    // launch shape: one persistent CTA per SM; the unit walk stride (CTAs, or pairs) is a multiple of n_ktiles so that a
    // CTA keeps its channel tile
    const int walkers_max = p.pair ? ctx->sm_count / 2 : ctx->sm_count;
    const int walk_units = p.pair ? p.total_units / 2 : p.total_units;
    int walkers = walkers_max < walk_units ? walkers_max : walk_units;
    walkers -= walkers % p.n_ktiles;
    if (walkers < p.n_ktiles) walkers = p.n_ktiles;
    const int grid = p.pair ? 2 * walkers : walkers;
    const int units_per_cta = (walk_units + walkers - 1) / walkers;

    // Full-halo plan (3x3, stride 1, 64-channel k-blocks, images of at least 8 x 16 pixels, filter bank resident): tiles
    // of 8 x 16 pixels, one framed box per channel block serves all nine taps, so the input crosses L2 -> SM once
    // (three times with vertical tap reuse, nine without) and a ring slot holds a whole channel block of a unit.
    // (up to 128 channels per tile: wider tiles share a unit between the issuing threads, which full-halo stages do not do)
    const bool fh_ok = n_tile <= 128 && R == 3 && pb.stride == 1 && n_par == 1 && pb.ic % 64 == 0 && gw >= 8 && gh >= 16 && ctx->use_full_halo &&
                       9 * (pb.ic / 64) * b_rows * 64 * 2 <= (p.pair ? 148 : 96) * 1024;
    // shared-memory plan.  Preference: haloed stages (vertical tap reuse) with 64-channel k-blocks, then with
    // 32-channel k-blocks (smaller stages, so that a ring of at least four still fits), else one tap per stage.
    const int ring_budget = 217 * 1024;   // 227 KB per CTA less the static arrays (8.3 KB) and the alignment slack
    const int kb_natural = (pb.ic % 64 == 0) ? 64 : (pb.ic % 32 == 0) ? 32 : 16;
    const bool can_vreuse = (R == 3 && pb.stride == 1 && p.bn == 1);
    const int taps_total = R * R;
    const int attempts[3][2] = {{kb_natural, 1}, {32, 1}, {kb_natural, 0}};   // (kb, vreuse)
    bool planned = false;
    // Merged horizontal taps (3x3, stride 1, one channel tile of 64, 64-channel k-blocks, image rows of 8 / 16 / 32 pixels that
    // fill a tile with whole rows): per vertical tap and k-step ONE MMA with N = 192 against the three filter columns, so
    // the A operand crosses the shared-memory port once per 192 columns instead of once per 64 (an N = 64 MMA is bound by
    // its operand fetch: 48 cycles for 32 cycles of tensor work).  The stage is the tile with a halo row above and below
    // (vertical taps are row offsets, as with vertical tap reuse); the horizontal shifts are applied to the three column
    // blocks of the accumulator by the epilogue.
    const bool hm_ok = ctx->use_hmerge && !p.pair && R == 3 && pb.stride == 1 && n_par == 1 && n_tile == 64 && pb.oc == 64 && pb.ic % 64 == 0 && !pb.out_f32 &&
                       pb.bias == nullptr && (gw == 8 || gw == 16 || gw == 32) && gh >= 128 / gw && 9 * pb.ic * 64 * 2 <= 148 * 1024;
    if (hm_ok && units_per_cta >= 2) {
        const int bank = 9 * pb.ic * 64 * 2;
        p.bw = gw; p.bh = 128 / gw; p.bn = 1;
        p.tiles_w = 1; p.tiles_h = gh / p.bh; p.tiles_n = pb.n;
        p.total_units = p.tiles_n * p.tiles_h * p.n_ktiles;
        const int a_bytes = (p.bh + 2) * p.bw * 128;   // multiples of 1 KB for every row length used here
        // Five slots and the blocks of the epilogue beat six slots (a data gradient of 50 images loses 0.5 us, but the forward pass gains, and a
        // program that runs both loads one kernel less: a kernel that comes to the SMs from DRAM costs about 5 us)
        int stages = (ring_budget - bank - 16 * 1024) / a_bytes;
        if (stages < 3) stages = (ring_budget - bank) / a_bytes;
        if (stages > kMaxStages) stages = kMaxStages;
        if (stages >= 3) {
            p.hm = 1; p.fh = 0; p.vreuse = 0; p.pair = 0;
            p.kb = 64; p.c_blocks = pb.ic / 64; p.swz = SWZ_128B;
            p.nb = 3; p.b_merged = 1;
            p.tx_b = 3 * 64 * 64 * 2; p.b_bytes = p.tx_b;          // one tile = the three filter columns of one filter row: 192 rows of 128 bytes
            p.tx_a = a_bytes; p.a_bytes = a_bytes; p.a_step = p.bw * 128;   // one image row per vertical tap
            p.resident = 1; p.resident_bytes = bank;
            p.stages = stages;
            p.acc_cols = 192; p.acc_bufs = 2; p.acc_shift = 1; p.tmem_cols = 512;
            planned = true;
        }
    }
    // (a pair's bank of 147 KB takes six units to pay: 128 -> 128 at 16x16 with 128 images, two units, 15.7 us, 13.7 without; with
    // 384, six units, 25.8 and 25.4 forward, 25.8 and 26.7 backward; with 1024 55.1 and 60.9)
    if (!planned && fh_ok && units_per_cta >= (9 * (pb.ic / 64) * b_rows * 128 > 96 * 1024 ? 6 : 2)) {
        const int tx_b = b_rows * 64 * 2, bank = taps_total * (pb.ic / 64) * tx_b, a_bytes = ((10 * 18 * 128) + 1023) & ~1023;
        int stages = (ring_budget - bank) / a_bytes;
        if (stages > kMaxStages) stages = kMaxStages;
        if (stages >= (p.pair ? 2 : 3)) {
            p.bw = 8; p.bh = 16; p.bn = 1;
            p.tiles_w = gw / 8; p.tiles_h = gh / 16; p.tiles_n = pb.n;
            p.fh = 1; p.vreuse = 0;
            p.kb = 64; p.c_blocks = pb.ic / 64; p.swz = SWZ_128B;
            p.tx_b = tx_b; p.b_bytes = tx_b; p.b_merged = 1; p.nb = 3;   // bank order [s][cb][r], three filter rows per load
            p.tx_a = 10 * 18 * 128; p.a_bytes = a_bytes; p.a_step = 0;
            p.resident = 1; p.resident_bytes = bank;
            p.stages = stages;
            planned = true;
        }
    }
    for (int a = 0; a < 3 && !planned; ++a) {
        const int kb = attempts[a][0], vr = attempts[a][1];
        if (vr && !can_vreuse) continue;
        if (kb > kb_natural) continue;
        p.kb = kb;
        p.c_blocks = pb.ic / kb;
        p.swz = kb == 64 ? SWZ_128B : kb == 32 ? SWZ_64B : SWZ_32B;
        p.vreuse = vr;
        p.tx_b = b_rows * kb * 2;
        p.b_merged = (vr && p.tx_b % 1024 == 0) ? 1 : 0;   // tiles of one load lie back to back: they must keep the swizzle alignment
        p.b_bytes = (p.tx_b + 1023) & ~1023;
        const int a_rows = vr ? (p.bh + 2) * p.bw : 128;
        p.tx_a = a_rows * kb * 2;
        p.a_bytes = (p.tx_a + 1023) & ~1023;
        p.nb = vr ? 3 : 1;
        p.a_step = vr ? p.bw * kb * 2 : 0;
        // (a pair could keep its half of a 3x3x128x128 bank, 148 KB, resident; measured slower than streaming it: the
        // ring left over is short)
        const int bank_bytes = taps_total * p.c_blocks * p.b_bytes;
        p.resident = (n_par == 1 && bank_bytes <= 96 * 1024 && units_per_cta >= 2) ? 1 : 0;
        p.resident_bytes = p.resident ? bank_bytes : 0;
        const int stage_bytes = p.a_bytes + (p.resident ? 0 : p.nb * p.b_bytes);
        int stages = (ring_budget - p.resident_bytes) / stage_bytes;
        if (stages > kMaxStages) stages = kMaxStages;
        p.stages = stages;
        if (stages >= 4 || !vr) break;
    }
    if (p.stages < 2) return B2C_ERR_UNSUPPORTED_SHAPE;
    int cluster = 0;   // CTAs per cluster of a split-K plan
    if (ctx->use_split_k && units_per_cta <= 2) {
        const int max_taps = n_par > 1 ? ((R + 1) / 2) * ((R + 1) / 2) : taps_total;
        const int a_rows = p.vreuse ? (p.bh + 2) * p.bw / 3 : p.fh ? 180 / 9 : 128;
        ConvKParams q = p;
        q.bw = gw < 128 ? gw : 128; q.bh = (128 / q.bw) < gh ? (128 / q.bw) : gh; q.bn = 128 / (q.bw * q.bh);
        q.tiles_w = gw / q.bw; q.tiles_h = gh / q.bh; q.tiles_n = (pb.n + q.bn - 1) / q.bn;
        q.vreuse = q.fh = q.hm = q.resident = q.resident_bytes = q.b_merged = q.a_step = 0;
        const int block = kblock_cycles(n_tile, p.kb, p.pair != 0, a_rows);
        const int least = kb_natural < 64 ? (p.vreuse ? 490 : 900) : p.vreuse ? 0 : 400, per_block = block > least ? block : least;
        const bool reuse = p.vreuse || p.fh || p.hm;   // taps share their loads
        const long long persistent = (long long)units_per_cta * max_taps * (pb.ic / p.kb) * per_block + 1060ll * n_tile / 32 +
                                     (p.pair ? 2600 : !reuse && units_per_cta > 1 ? 3000 : 0);
        if (choose_splitk(ctx, pb, q, n_par * m_tiles, reuse, persistent)) {
            p = q;
            cluster = p.splits * (p.pair ? 2 : 1);
            b_rows = p.pair ? p.n_tile / 2 : p.n_tile;
        }
    }
    p.mma_n = p.hm ? 3 * p.n_tile : p.n_tile;
    // Short k-blocks share a ring slot.  An issuing thread pays 700-900 cycles per slot on top of its MMAs (the slot's stamp,
    // the barrier wait, two commits; measured inside the running kernel), which bounds the stride-2 and 1x1 layers
    // (one k-block = 2-4 MMAs of 48-128 cycles): group k-blocks while a slot holds less than about 1000 tensor-pipe
    // cycles, three slots remain (four where two threads take alternate slots) and the unit has that many k-blocks.
    if (!cluster) p.gsub = 1;
    if (ctx->use_group_kblocks && !cluster && !p.fh && !p.hm && !p.vreuse) {
        // k-blocks of the longest unit (stride-2 data gradient: the parity that takes every other tap in both directions)
        const int max_sub = (n_par > 1 ? ((R + 1) / 2) * ((R + 1) / 2) : taps_total) * p.c_blocks;
        const int per_sub = (p.kb / 16) * (p.mma_n / 2 > 48 ? p.mma_n / 2 : 48);
        const bool split = p.n_tile > 128 && ctx->use_issue_split;   // two threads on alternate slots: an even ring, and four slots so that each keeps two
        int g = 1;
        while (g < 4 && g * per_sub < 1000 && 2 * g <= max_sub) {
            int slots = p.stages / (2 * g);
            if (split) slots &= ~1;
            if (slots < (split ? 4 : 3)) break;
            g *= 2;
        }
        p.gsub = g;
        p.stages /= g;
    }
    // Two issuing threads where one cannot keep the tensor pipe busy: tiles of at most 128 channels.
    p.issuers = p.n_tile <= 128 ? kIssuers : 1;
    // Wider tiles: both threads work on every unit, alternate stages (needs an even ring).
    if (!cluster && p.n_tile > 128 && ctx->use_issue_split && p.stages >= 2) {
        p.stages &= ~1;
        p.issuers = kIssuers;
        p.issue_split = 1;
    }
    const int stage_bytes = p.gsub * (p.a_bytes + (p.resident ? 0 : p.nb * p.b_bytes));
    // Epilogue in blocks, where shared memory has room for them beside the ring (a shorter ring costs more than they give: 256 -> 1024 1x1 at
    // 8x8 59 -> 64 us): tiles of 64 channels 32 columns at a time; 128 and 256 channels 64 at a time, full-halo stages, which leave no room,
    // 16 at a time in the kernel's static arrays.  Tiles of 256 channels without sums whose MMAs take more than 12000 cycles hide the
    // epilogue anyway and are 1 % slower in blocks (256 -> 256 at 8x8 59.7 and 60.1 us), and so are 64-channel tiles with vertical tap reuse in
    // k-blocks of 32 channels from 5000 cycles on, or with one k-block, no sums and more than two units per CTA (rows / blocks at 32x32: 608 -> 64 with 60 images without sums
    // 94.6 and 97.4 us, 224 -> 64 with 150 69.1 and 70.8, with sums 70.6 and 72.4, 160 -> 64 with 200 63.3 and 63.4, with sums 64.6 and 64.9; 32 ->
    // 64 with 500 35.9 and 37.4, but with sums 38.7 and 37.5, and with 4 at 64x64, one unit each, 6.6 and 6.2); the others gain, see epilogue_blocks.  Large 1x1 layers without sums that move as
    // much in as out are bound by HBM and differ by what else is in flight: 64 -> 64 at 32x32 with 1024 images on its own 47.0 by rows and 50.5
    // in blocks, as a data gradient inside a step 59 and 51.
    if (!cluster && !pb.out_f32 && pb.bias == nullptr) {
        const bool sums = (pb.stats != nullptr || pb.ask_sums) && pb.bwd_y == nullptr;
        const int room = ring_budget - p.resident_bytes - p.stages * stage_bytes;
        const int mma = R * R * pb.ic / 16 / n_par * (n_tile / 2);
        const bool hidden = p.vreuse && p.kb == 32 && (R * R * pb.ic / 16 * 48 >= 5000 || (!sums && p.c_blocks == 1 && units_per_cta > 2));
        if (n_tile == 64 && !p.fh && !hidden && room >= 16 * 1024) p.block_cols = 32;
        if (n_tile == 128) p.block_cols = p.fh ? 16 : room >= 24 * 1024 ? 64 : 0;
        if (n_tile == 256 && p.issue_split && room >= 24 * 1024 && (sums || mma < 12000)) p.block_cols = 64;
    }
    const int block_bytes = p.block_cols == 64 ? 24 * 1024 : p.block_cols == 32 ? 16 * 1024 : 0;
    size_t smem_bytes = (size_t)p.resident_bytes + (size_t)p.stages * stage_bytes + 1024 +
                        block_bytes + (cluster && !p.x_overlap ? (size_t)(p.splits - 1) * (p.n_tile / p.splits) * 512 : 0);
    // CTAs that wait for one another (pairs, and clusters that share a tile) take more than half of an SM's shared memory, so that no two of
    // them share an SM.  Their TMEM allocations wait for columns without a limit: two clusters of different streams (or three) that met on
    // several SMs could each hold the columns that the other one's partner waits for.
    if ((p.pair || p.splits > 1) && smem_bytes < kClusterSmem) smem_bytes = kClusterSmem;

    plan.grid = cluster ? p.total_units * p.splits : grid;
    plan.smem_bytes = smem_bytes;
    if (pb.in == nullptr) return B2C_OK;   // a question about the plan

    // tensor maps
    const int box_h = (p.vreuse || p.fh || p.hm) ? p.bh + 2 : p.bh;
    const int box_w = p.fh ? p.bw + 2 : p.bw;
    if (!pb.dgrad && pb.stride == 2) {
        for (int ph = 0; ph < 2; ++ph)
            for (int pw = 0; pw < 2; ++pw)
                if (!encode_activation_map(ctx, &p.tmA[ph * 2 + pw], pb.in, pb.n, pb.ih, pb.iw, pb.ic, 2, ph, pw, p.kb, box_w, box_h, p.bn))
                    return B2C_ERR_CUDA;
    } else {
        if (!encode_activation_map(ctx, &p.tmA[0], pb.in, pb.n, pb.ih, pb.iw, pb.ic, 1, 0, 0, p.kb, box_w, box_h, p.bn)) return B2C_ERR_CUDA;
    }
    if (p.hm) {
        // weights [out][r][s][in] viewed as (in, out, s, r): a box of all nine taps lands as [r][s][out][in], i.e. per filter row
        // one K-major tile whose 192 rows are the three filter columns of the 64 output channels
        cuuint64_t dims[4] = {(cuuint64_t)pb.ic, (cuuint64_t)pb.oc, (cuuint64_t)R, (cuuint64_t)R};
        cuuint64_t str[3] = {(cuuint64_t)R * R * pb.ic * 2, (cuuint64_t)pb.ic * 2, (cuuint64_t)R * pb.ic * 2};
        cuuint32_t box[4] = {64u, 64u, 3u, 3u};
        if (!encode_map(ctx, &p.tmB, pb.wt, 4, dims, str, box, 128)) return B2C_ERR_CUDA;
    } else {
        // weights [out][r][s][in] viewed as (in, s, out, r): a box of three filter rows lands as three tiles [r][out][in]
        cuuint64_t dims[4] = {(cuuint64_t)pb.ic, (cuuint64_t)R, (cuuint64_t)pb.oc, (cuuint64_t)R};
        cuuint64_t str[3] = {(cuuint64_t)pb.ic * 2, (cuuint64_t)R * R * pb.ic * 2, (cuuint64_t)R * pb.ic * 2};
        cuuint32_t box[4] = {(cuuint32_t)p.kb, 1u, (cuuint32_t)b_rows, p.b_merged ? 3u : 1u};
        if (!encode_map(ctx, &p.tmB, pb.wt, 4, dims, str, box, p.kb * 2)) return B2C_ERR_CUDA;
    }

    // tap tables (row-major over (r, s); with vreuse entry s of row 0 carries the shift of the haloed tile)
    if (!pb.dgrad) {
        forward_taps(p.taps[0], R, pb.stride, pb.pad);
        p.os_n = (long long)pb.oh * pb.ow * pb.oc; p.os_h = (long long)pb.ow * pb.oc; p.os_w = pb.oc;
    } else if (pb.stride == 1) {
        TapList& tl = p.taps[0];
        for (int r = 0; r < R; ++r)   // r, s index the flipped filter
            for (int s = 0; s < R; ++s) {
                const int i = tl.count++;
                tl.map[i] = 0; tl.dh[i] = (int8_t)(r - (R - 1 - pb.pad)); tl.dw[i] = (int8_t)(s - (R - 1 - pb.pad));
                tl.rs[i] = (int8_t)(r * R + s);
            }
        p.os_n = (long long)pb.oh * pb.ow * pb.oc; p.os_h = (long long)pb.ow * pb.oc; p.os_w = pb.oc;
    } else {
        for (int ph = 0; ph < 2; ++ph)
            for (int pw = 0; pw < 2; ++pw) {
                TapList& tl = p.taps[ph * 2 + pw];
                for (int rf = 0; rf < R; ++rf)
                    for (int sf = 0; sf < R; ++sf) {
                        const int r = R - 1 - rf, s = R - 1 - sf;   // tap of the forward filter
                        const int eh = ph + pb.pad - r, ew = pw + pb.pad - s;
                        if ((eh & 1) || (ew & 1)) continue;
                        const int i = tl.count++;
                        tl.map[i] = 0; tl.dh[i] = (int8_t)(eh / 2); tl.dw[i] = (int8_t)(ew / 2);
                        tl.rs[i] = (int8_t)(rf * R + sf);
                    }
                p.off[ph * 2 + pw] = ((long long)ph * pb.ow + pw) * pb.oc;
            }
        p.os_n = (long long)pb.oh * pb.ow * pb.oc; p.os_h = 2ll * pb.ow * pb.oc; p.os_w = 2ll * pb.oc;
    }
    for (int i = 0; i < 7; ++i) {
        const int v = 1 << i;
        p.row_bit[i] = (int)(v < p.bw ? p.os_w * v : v < p.bw * p.bh ? p.os_h * (v / p.bw) : p.os_n * (v / (p.bw * p.bh)));
    }
    p.r_filter = R;
    p.n_valid = pb.n;
    p.oc_valid = pb.oc;
    p.out = pb.out;
    p.out_is_f32 = pb.out_f32 ? 1 : 0;
    p.out_v8 = (reinterpret_cast<uintptr_t>(pb.out) % 32 == 0) ? 1 : 0;   // row pitches are multiples of 32 bytes (16 channels)
    p.bias = pb.bias;
    p.stats = pb.out_f32 ? nullptr : pb.stats;
    p.stats_group_images = pb.stats_group_images;
    p.tw_shift = log2_exact(p.tiles_w);
    p.th_shift = log2_exact(p.tiles_h);
    p.nk_shift = log2_exact(p.n_ktiles);
    p.grp_shift = log2_exact(p.stats_group_images);
    p.cb_shift = log2_exact(p.c_blocks);
    // Sums of a BatchNorm's backward pass: the one-wave kernel only, whose layers are bound by launches.  In the persistent kernel the other
    // operands' latency comes once per unit: 64 -> 64 3x3 with 1024 images 66 -> 140 us for 45 us less in the BatchNorm.
    if (pb.bwd_y != nullptr && (!cluster || (p.stats_group_images > 0 && p.stats_group_images % p.bn != 0))) p.stats = nullptr;
    if (p.stats && p.stats_group_images > 0 && (p.stats_group_images % p.bn) != 0) return B2C_ERR_UNSUPPORTED_SHAPE;  // a tile must not straddle groups
    return B2C_OK;
}

static int kernel_kind(const ConvKParams& p) { return p.hm ? KIND_HMERGE : p.fh ? KIND_FULL_HALO : p.issue_split ? KIND_SPLIT : KIND_GENERAL; }

bool kmajor_sums_in_blocks(b2c_ctx* ctx, KMajorProblem pb)
{
    pb.in = pb.wt = pb.out = nullptr;
    pb.stats = nullptr;
    pb.ask_sums = true;
    KMajorPlan plan;
    return build_kmajor_plan(ctx, pb, plan) == B2C_OK && plan.p.block_cols != 0;
}

b2c_status plan_conv_kmajor(b2c_ctx* ctx, const KMajorProblem& pb, b2c_conv_plan_detail& detail)
{
    static_assert((int)KIND_GENERAL == B2C_PLAN_GENERAL && (int)KIND_SPLIT == B2C_PLAN_SHARED_UNITS && (int)KIND_HMERGE == B2C_PLAN_MERGED_TAPS &&
                      (int)KIND_FULL_HALO == B2C_PLAN_FULL_HALO, "the header's names of the kernel kinds");
    KMajorPlan plan;
    b2c_status st = build_kmajor_plan(ctx, pb, plan);
    if (st != B2C_OK) return st;
    const ConvKParams& p = plan.p;
    b2c_conv_plan& out = detail.plan;
    out.kind = p.splits > 0 ? B2C_PLAN_ONE_WAVE : kernel_kind(p);
    out.tile_channels = p.n_tile; out.pair = p.pair; out.splits = p.splits > 0 ? p.splits : 1; out.overlap = p.x_overlap;
    out.ctas = plan.grid; out.smem_bytes = (int)plan.smem_bytes;
    out.k_block = p.kb; out.slot_k_blocks = p.gsub;
    detail.block_cols = p.block_cols;
    return B2C_OK;
}

b2c_status launch_conv_kmajor(b2c_ctx* ctx, const KMajorProblem& pb, cudaStream_t stream)
{
    // plans are keyed by everything the planner reads: the problem and the context's switches
    const int switches = ctx->use_pairs | ctx->use_full_halo << 4 | ctx->use_issue_split << 5 | ctx->use_hmerge << 6 | ctx->use_group_kblocks << 7 | ctx->use_split_k << 8;
    const b2c_plan_key key = {{b2c_key_pair('K', switches), b2c_key_pair(pb.n, pb.stats_group_images), b2c_key_pair(pb.ih, pb.iw), b2c_key_pair(pb.oh, pb.ow),
                               b2c_key_pair(pb.ic, pb.oc), b2c_key_pair(pb.r, pb.stride), b2c_key_pair(pb.pad, pb.dgrad | pb.out_f32 << 1 | (pb.bwd_y != nullptr) << 2), b2c_key_ptr(pb.in),
                               b2c_key_ptr(pb.wt), b2c_key_ptr(pb.out), b2c_key_ptr(pb.bias), b2c_key_ptr(pb.stats)}};
    auto it = ctx->plan_cache.find(key);
    if (it == ctx->plan_cache.end()) {
        KMajorPlan fresh;
        b2c_status st = build_kmajor_plan(ctx, pb, fresh);
        if (st != B2C_OK) return st;
        if (ctx->plan_cache.size() >= 8192) ctx->plan_cache.clear();   // callers that pass new buffers every call: keep the table bounded
        std::vector<unsigned char> bytes(sizeof(KMajorPlan));
        memcpy(bytes.data(), &fresh, sizeof(KMajorPlan));
        it = ctx->plan_cache.emplace(key, std::move(bytes)).first;
    }
    KMajorPlan plan;   // a copy: the 64-byte alignment of the tensor maps is the parameter block's, not the table's
    memcpy(&plan, it->second.data(), sizeof(KMajorPlan));
    ConvKParams& p = plan.p;
    const int grid = plan.grid;
    const size_t smem_bytes = plan.smem_bytes;
    p.no_wait = pb.no_wait ? 1 : 0;
    const bool bwd = pb.bwd_y != nullptr && p.stats != nullptr;
    p.bwd_y = bwd ? pb.bwd_y : nullptr;
    p.bwd_other = pb.bwd_other;
    p.bwd_mask = reinterpret_cast<const uint8_t*>(pb.bwd_mask);
    if (pb.bwd_done != nullptr) *pb.bwd_done = bwd;
    p.status = ctx->d_status;
    p.spin_limit = ctx->spin_limit;
    p.stall = ctx->stall_counters;

    if (p.splits > 0) return launch_conv_splitk(ctx, p, grid, smem_bytes, stream);
    // the kernel kind of the plan (merged taps run on single CTAs only)
    typedef void (*kernel_t)(const ConvKParams);
    static const kernel_t kernels[2][2][4] = {
        {{conv_kmajor_kernel<false, KIND_GENERAL, false>, conv_kmajor_kernel<false, KIND_SPLIT, false>, conv_kmajor_kernel<false, KIND_HMERGE, false>,
          conv_kmajor_kernel<false, KIND_FULL_HALO, false>},
         {conv_kmajor_kernel<true, KIND_GENERAL, false>, conv_kmajor_kernel<true, KIND_SPLIT, false>, nullptr, conv_kmajor_kernel<true, KIND_FULL_HALO, false>}},
        // (128-channel tiles: the filter bank of a full-halo plan fits only halved, for a pair)
        {{conv_kmajor_kernel<false, KIND_GENERAL, true>, conv_kmajor_kernel<false, KIND_SPLIT, true>, conv_kmajor_kernel<false, KIND_HMERGE, true>, nullptr},
         {conv_kmajor_kernel<true, KIND_GENERAL, true>, conv_kmajor_kernel<true, KIND_SPLIT, true>, nullptr, conv_kmajor_kernel<true, KIND_FULL_HALO, true>}}};
    const kernel_t kernel = kernels[p.block_cols ? 1 : 0][p.pair ? 1 : 0][kernel_kind(p)];
    if (kernel == nullptr) return B2C_ERR_UNSUPPORTED_SHAPE;
    if (!(ctx->smem_optin_done & B2C_OPTIN_KMAJOR)) {   // the attribute belongs to the device: kept per context, not per process
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
                if (kernels[a >> 1][a & 1][b] != nullptr)
                    B2C_CUDA(cudaFuncSetAttribute(kernels[a >> 1][a & 1][b], cudaFuncAttributeMaxDynamicSharedMemorySize, 218 * 1024));
        ctx->smem_optin_done |= B2C_OPTIN_KMAJOR;
    }
    B2C_CUDA(b2c_launch(ctx, kernel, dim3((unsigned)grid), dim3(kThreads), smem_bytes, stream, p.pair ? 2u : 1u, p));
    B2C_CUDA(cudaGetLastError());
    return B2C_OK;
}

}  // namespace b2c
