// The direct 3x3 convolution (stride 1 or 2, pad 1) as ONE implicit GEMM on the tcgen05 tensor cores:
//     y[k][p] = sum over taps (dy, dx) and channels c of  w[tap][k][c] * x[c][p shifted by the tap].
// direct_pack_kernel writes x once more with 8 channels of a pixel side by side (16-byte pieces) and zeros between the
// image rows; the convolution kernel brings a patch of it with its halo into shared memory once per (tile of pixels, 64
// input channels), and the nine taps are then nine START ADDRESSES into that patch.  Neither the nine shifted copies of x
// nor the per-tap products of the three-step form exist.
//
// Operand A (pixels, UMMA M = 128 lanes): K-major WITHOUT swizzle, i.e. for every 8 channels one array of 16-byte
// pieces, one per pixel position of the patch.  A row of the operand is one piece, eight consecutive rows are 128
// contiguous bytes, groups of eight rows are SBO apart and the next 8 channels are LBO apart, so moving the operand by
// one pixel is adding 16 bytes to the start address, and by one image row adding `pitch` pieces.
// Two ways to lay pixels on the 128 lanes:
//   grid: 16 output rows x 8 output columns; groups of eight lanes = eight columns of one row, SBO = one patch row;
//   flat: 128 consecutive positions of the image read row by row with ONE column and one row of zeros between
//         neighbours (the right padding of a row is the left padding of the next); SBO = 128 bytes.  Positions that
//         fall on the padding are computed and dropped, 1 / (W + 1) of the work, where a grid would hang over the
//         edges of a ragged or small image by more than that.
// With stride 2 the patch is four patches, one per parity of (row, column): every tap reads one of them.
// Operand B (filters, UMMA N = n_tile output channels): the blocked taps U[9][Cb][Kb][16][64] by TMA, 128-byte swizzle.
//
// A CTA owns 128 pixels x n_tile output channels (two sets of fp32 accumulators in TMEM, so that the epilogue of a tile
// overlaps the next) and walks all channels, or one of `splits` parts of them: layers with few pixels have too few tiles
// for 148 SMs otherwise.  The parts then go to the workspace in fp32 and direct_reduce_kernel adds them in a fixed order.
// (256 pixels per CTA tile, the filter box used twice, was slower on all of 24 layers: it leaves half as many CTAs and
// two stages for the patches.)
// What bounds it: the MMAs of a tap, 52 cycles each or n_tile / 2, and some 30 cycles around them; without the loads it
// takes as long within 5 %.
// Against the three steps (times in us, one layer in a graph): stride 2, 320 -> 320 at 64x64, batch 2: 20.0 -> 14.7; at
// 96x96, batch 4: 73.0 -> 32.2; at 113x89, batch 2: 42.4 -> 28.3; 640 -> 640 at 64x64, batch 2: 40 -> 26.9; stride 1,
// 640 -> 640 at 32x32, batch 2: 39.6 -> 20.5; 1280 -> 1280 at 8x8, batch 8: 26.7 -> 24.2.
//   warp 0      filter producer (TMA)         warps 2-9   epilogue (two per TMEM lane quarter)
//   warp 1      TMEM owner and MMA issuer     warp 10     patch producer (TMA)
#pragma once
#include <cuda_fp16.h>

#include "ptx.cuh"
#include "transforms.cuh"
#include "wino_gemm.cuh"

namespace sdw {

constexpr int DC_EPI_WARPS = 8;
constexpr int DC_THREADS = (2 + DC_EPI_WARPS + 1) * 32;
constexpr int DC_EPI_CH = 8;              // output channels a warp stages at a time
constexpr int DC_STG_BYTES = DC_EPI_CH * 32 * 4;
constexpr int DC_MAX_A_STAGES = 6;
constexpr int DC_MAX_B_STAGES = 16;
constexpr int DC_BARS = 2 * DC_MAX_A_STAGES + 2 * DC_MAX_B_STAGES + 4;
constexpr int DC_BAR_BYTES = DC_BARS * 8 + 16;

struct DirectParams {
    const uint32_t* wt_header;
    const __half* x;
    const __half* bias;
    const __half* residual;
    __half* y;
    const __half* packed;     // see direct_pack_kernel
    float* part;              // splits > 1: fp32 parts [(pixel tile, k tile)][split][n_tile][128]
    int act;
    int N, C, H, W, K, Ho, Wo, stride; // N: images of this launch; x, y and residual point at its first output
    int n_tile, num_k_tiles, num_m;    // output channels per CTA tile, tiles along k and along the pixels
    int pair_begin, pair_end;          // (pixel tile, k tile) pairs of this launch
    int splits, cb_per_split, num_cb;  // parts of the channel blocks
    int flat, pitch, rows_img;         // layout of the pixels; rows_img: rows per image, padding included
    int lead;                          // flat, stride 1: positions of zeros before the first pixel
    int tiles_c, tiles_r;              // grid: tiles per image
    int PP;                            // pixel positions of a patch (one plane of it)
    int planes;                        // 1, or 4 with stride 2
    int sbo;                           // 16-byte pieces between groups of eight lanes
    int pk_pitch, pk_pieces;           // packed copy: row pitch (positions) and 8-channel pieces per plane
    long long pk_positions;            // its positions per piece
    int vec_store;                     // grid: rows of eight outputs are aligned 16-byte pieces of y (and residual)
    int a_stage_bytes, a_stages, b_stages;
    FastDiv fd_pitch, fd_rows, fd_k, fd_s, fd_tc, fd_tr, fd_pkp;
    // (last: between the fields above, which the convolution kernel reads, they cost a launch of 14 us 0.1 us)
    int win_h, win_w;                  // output rows and columns of this launch (all, unless the workspace is small)
    int row0, col0;                    // row and column of x at position (0, 0) of the packed copy
};

// No swizzle, K-major: [0,14) start >> 4, [16,30) bytes between 8-channel pieces >> 4, [32,46) bytes between groups of
// eight rows >> 4, [46,48) version 1.
__device__ __forceinline__ uint64_t make_smem_desc_plain(uint32_t smem_addr, uint32_t lbo_units, uint32_t sbo_units) {
    return static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(lbo_units & 0x3FFFu) << 16) |
           (static_cast<uint64_t>(sbo_units & 0x3FFFu) << 32) | (static_cast<uint64_t>(1) << 46);
}

// The order of the nine taps: with stride 2 those of one plane follow one another.
template <int STRIDE> __host__ __device__ constexpr int direct_tap(int t) {
    constexpr int by_plane[9] = {0, 2, 6, 8, 1, 7, 3, 5, 4};
    return STRIDE == 1 ? t : by_plane[t];
}
template <int STRIDE> __host__ __device__ constexpr bool direct_first_of_plane(int t) {
    return t == 0 || (STRIDE == 2 && (t == 4 || t == 6 || t == 8));
}

// PART: the launch covers part of the rows or columns.  A flag of its own: the two further parameters that the epilogue then
// reads cost a launch on whole images 0.1 us.
template <bool PART> __device__ __forceinline__ int direct_win_h(const DirectParams& q) { return PART ? q.win_h : q.Ho; }
template <bool PART> __device__ __forceinline__ int direct_win_w(const DirectParams& q) { return PART ? q.win_w : q.Wo; }

// Lane `l` (0..127) of CTA tile m -> image, output row and column; false where nothing is stored.
template <bool PART>
__device__ __forceinline__ bool direct_out_pixel(const DirectParams& q, int m, int l, int& n, int& r, int& c) {
    if (q.flat) {
        const uint32_t Q = static_cast<uint32_t>(m) * 128u + static_cast<uint32_t>(l);
        const uint32_t v = fast_div(Q, q.fd_pitch);
        c = static_cast<int>(Q - v * static_cast<uint32_t>(q.pitch));
        const uint32_t img = fast_div(v, q.fd_rows);
        r = static_cast<int>(v - img * static_cast<uint32_t>(q.rows_img));
        n = static_cast<int>(img);
        return n < q.N && r < direct_win_h<PART>(q) && c < direct_win_w<PART>(q);
    }
    const uint32_t row_blk = fast_div(static_cast<uint32_t>(m), q.fd_tc);
    const uint32_t img = fast_div(row_blk, q.fd_tr);
    const int cb = m - static_cast<int>(row_blk) * q.tiles_c;
    const int rb = static_cast<int>(row_blk) - static_cast<int>(img) * q.tiles_r;
    n = static_cast<int>(img);
    r = rb * 16 + (l >> 3);
    c = cb * 8 + (l & 7);
    return r < direct_win_h<PART>(q) && c < direct_win_w<PART>(q);
}

template <int STRIDE, bool PART>
__global__ void __launch_bounds__(DC_THREADS, 1)
direct_conv_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmX,
                   const __grid_constant__ DirectParams q, int* __restrict__ status_word) {
    extern __shared__ uint8_t dc_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dc_smem_raw) + 1023) & ~uintptr_t(1023));
    const int b_stage_bytes = q.n_tile * 128;
    uint8_t* a_base = smem + q.b_stages * b_stage_bytes;
    float* stg_base = reinterpret_cast<float*>(a_base + q.a_stages * q.a_stage_bytes);
    uint64_t* b_full = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(stg_base) + DC_EPI_WARPS * DC_STG_BYTES);
    uint64_t* b_empty = b_full + DC_MAX_B_STAGES;
    uint64_t* a_full = b_empty + DC_MAX_B_STAGES;
    uint64_t* a_empty = a_full + DC_MAX_A_STAGES;
    uint64_t* acc_full = a_empty + DC_MAX_A_STAGES;
    uint64_t* acc_empty = acc_full + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (threadIdx.x < DC_BARS) {     // one thread per barrier, in the order of the pointers above
        mbar_init(&b_full[threadIdx.x], threadIdx.x >= DC_BARS - 2 ? DC_EPI_WARPS : 1);
        fence_barrier_init();
    }
    if (threadIdx.x == DC_THREADS - 32) {
        *abort_flag = 0;
        prefetch_tmap(&tmU);
        if (!q.flat) prefetch_tmap(&tmX);
    }
    if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
    pdl_launch_dependents();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const bool elected = elect_one() != 0;     // the single-threaded roles run as whole warps, this lane issues

    // The packing kernel waits for everything before it and then releases this one, so the filters are final here; the
    // packed x and y are not before the wait.
    const uint4 hdr = *reinterpret_cast<const uint4*>(q.wt_header);
    const bool wt_ok = hdr.x == WT_MAGIC && hdr.y == static_cast<uint32_t>(q.K) && hdr.z == static_cast<uint32_t>(q.C) &&
                       hdr.w == 1u;
    const int work_begin = q.pair_begin * q.splits, work_end = q.pair_end * q.splits;
    // work item -> (pixel tile m, k tile kt, first and last channel block)
    auto decode = [&](int wi, int& m, int& kt, int& cb0, int& cb1) {
        const uint32_t pair = fast_div(static_cast<uint32_t>(wi), q.fd_s);
        const int s = wi - static_cast<int>(pair) * q.splits;
        const uint32_t mm = fast_div(pair, q.fd_k);
        m = static_cast<int>(mm);
        kt = static_cast<int>(pair - mm * static_cast<uint32_t>(q.num_k_tiles));
        cb0 = s * q.cb_per_split;
        cb1 = min(cb0 + q.cb_per_split, q.num_cb);
    };

    if (!wt_ok) {
        pdl_wait();
        if (threadIdx.x == 0) atomicCAS(status_word, 0, 1 | (9 << 8));   // a filter buffer of another layer: nothing is read
    } else if (warp == 0) {
        // ------------------------------ filters ------------------------------
        const uint32_t base = smem_u32(smem), full0 = smem_u32(b_full), empty0 = smem_u32(b_empty);
        int stage = 0;
        uint32_t phase = 1, dst = base, bars = 0;      // bars: offset of the stage's barriers
        bool ok = true;
        for (int wi = work_begin + blockIdx.x; wi < work_end && ok; wi += gridDim.x) {
            int m, kt, cb0, cb1;
            decode(wi, m, kt, cb0, cb1);
            const int kb = (kt * q.n_tile) >> 4;
            for (int cb = cb0; cb < cb1 && ok; ++cb) {
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    ok = mbar_wait_warp_a32(empty0 + bars, &b_empty[stage], phase, abort_flag, GEMM_WAIT_LIMIT_NS);
                    if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 1, 0); break; }
                    if (elected) {
                        mbar_arrive_expect_tx_a32(full0 + bars, static_cast<uint32_t>(b_stage_bytes));
                        tma_load_5d_a32(dst, &tmU, full0 + bars, cb, kb, direct_tap<STRIDE>(t));
                    }
                    ++stage;
                    dst += b_stage_bytes;
                    bars += 8;
                    if (stage == q.b_stages) { stage = 0; dst = base; bars = 0; phase ^= 1u; }
                }
            }
        }
        if (!ok) *abort_flag = 1;
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        // What a tap costs beside its MMAs is what keeps the tensor pipe waiting, so the taps are unrolled with their offsets
        // known, descriptors and barriers only advance by additions and there is one way through the loop: a last block of
        // channels short of 64 is padded with zeros.  (With its k-steps counted, in the same loop or in one of its own, an
        // MMA cost 45-50 cycles of issue that nothing overlapped; 640 -> 640 at 32x32, batch 2, stride 2, 64 channels per
        // CTA and 90 taps: 21.4 us against 23.1-24.9.)
        const uint32_t idesc = make_idesc_f16_f32(128, q.n_tile, false, false);
        const uint64_t a_desc0 = make_smem_desc_plain(smem_u32(a_base), static_cast<uint32_t>(q.PP), static_cast<uint32_t>(q.sbo));
        const uint64_t b_desc0 = make_smem_desc_sw128(smem_u32(smem), 16, 1024);
        const uint64_t a_step = static_cast<uint64_t>(q.a_stage_bytes >> 4), b_step = static_cast<uint64_t>(b_stage_bytes >> 4);
        const uint64_t k_step = 2u * static_cast<uint64_t>(q.PP);       // 16 channels = two 8-channel arrays
        const uint64_t pitch = static_cast<uint64_t>(q.pitch);
        const uint32_t bfull0 = smem_u32(b_full), bempty0 = smem_u32(b_empty), afull0 = smem_u32(a_full), aempty0 = smem_u32(a_empty);
        int bs = 0, as = 0, buf = 0;
        uint64_t ad_stage = a_desc0, bd = b_desc0;
        uint32_t bbar = 0, abar = 0;                                    // offsets of the stages' barriers
        uint32_t bphase = 0, aphase = 0, acc_phase = 0;
        bool ok = true;
        for (int wi = work_begin + blockIdx.x; wi < work_end && ok; wi += gridDim.x) {
            int m, kt, cb0, cb1;
            decode(wi, m, kt, cb0, cb1);
            ok = mbar_wait_warp(&acc_empty[buf], acc_phase ^ 1u, abort_flag, GEMM_WAIT_LIMIT_NS);
            if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 2, 0); break; }
            tc_fence_after_sync();
            const uint32_t d0 = tmem_base + static_cast<uint32_t>(buf * q.n_tile);
            for (int cb = cb0; cb < cb1; ++cb) {
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    const int tap = direct_tap<STRIDE>(t);
                    const int dy = STRIDE == 1 ? tap / 3 : (tap / 3) >> 1, dx = STRIDE == 1 ? tap % 3 : (tap % 3) >> 1;
                    if (direct_first_of_plane<STRIDE>(t)) {
                        ok = mbar_wait_warp_a32(afull0 + abar, &a_full[as], aphase, abort_flag, GEMM_WAIT_LIMIT_NS);
                        if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 3, 0); break; }
                    }
                    ok = mbar_wait_warp_a32(bfull0 + bbar, &b_full[bs], bphase, abort_flag, GEMM_WAIT_LIMIT_NS);
                    if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 4, 0); break; }
                    tc_fence_after_sync();
                    const uint64_t ad = ad_stage + dy * pitch + dx;
                    const uint32_t acc = t > 0 || cb > cb0 ? 1u : 0u;
                    if (elected) {
                        umma_f16(d0, ad, bd, idesc, acc);
                        umma_f16_acc(d0, ad + k_step, bd + 2, idesc);
                        umma_f16_acc(d0, ad + 2 * k_step, bd + 4, idesc);
                        umma_f16_acc(d0, ad + 3 * k_step, bd + 6, idesc);
                    }
                    if (elected) umma_commit_a32(bempty0 + bbar);
                    ++bs;
                    bd += b_step;
                    bbar += 8;
                    if (bs == q.b_stages) { bs = 0; bd = b_desc0; bbar = 0; bphase ^= 1u; }
                    if (t == 8 || direct_first_of_plane<STRIDE>(t + 1)) {
                        if (elected) umma_commit_a32(aempty0 + abar);
                        ++as;
                        ad_stage += a_step;
                        abar += 8;
                        if (as == q.a_stages) { as = 0; ad_stage = a_desc0; abar = 0; aphase ^= 1u; }
                    }
                }
                if (!ok) break;
            }
            if (!ok) break;
            if (elected) umma_commit(&acc_full[buf]);
            buf ^= 1;
            if (buf == 0) acc_phase ^= 1u;
        }
        if (!ok) *abort_flag = 1;
    } else if (warp < 2 + DC_EPI_WARPS) {
        // ------------------------------ epilogue ------------------------------
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        pdl_wait();      // nothing is written before the predecessor has completed
        float* stg = stg_base + (warp - 2) * (DC_STG_BYTES / 4);
        const long long hw_o = static_cast<long long>(q.Ho) * q.Wo;
        int buf = 0;
        uint32_t acc_phase = 0;
        for (int wi = work_begin + blockIdx.x; wi < work_end; wi += gridDim.x) {
            int m, kt, cb0, cb1;
            decode(wi, m, kt, cb0, cb1);
            if (!mbar_wait_warp(&acc_full[buf], acc_phase, abort_flag, GEMM_WAIT_LIMIT_NS)) {
                if (lane == 0) { if (*abort_flag == 0) report_timeout(status_word, 5, 0); *abort_flag = 1; }
                break;
            }
            tc_fence_after_sync();
            const int k0 = kt * q.n_tile;
            if (q.splits == 1 && q.vec_store) {
                // The warp's 32 lanes are four rows of eight outputs.  DC_EPI_CH channels at a time go through shared memory
                // in fp32, [channel][32], and leave as 16-byte pieces: one lane per (channel, row).
                int n, oy, ox;
                direct_out_pixel<PART>(q, m, quarter * 32, n, oy, ox);
                const int row = lane & 3, ch = lane >> 2;
                for (int col = half * DC_EPI_CH; col < q.n_tile && k0 + col < q.K; col += 2 * DC_EPI_CH) {
                    uint32_t r[8];
                    tmem_ld_32x8_sync(tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                                      static_cast<uint32_t>(buf * q.n_tile + col), r);
#pragma unroll
                    for (int j = 0; j < DC_EPI_CH; ++j) stg[j * 32 + lane] = __uint_as_float(r[j]);
                    __syncwarp();
                    {
                        const int k = k0 + col + ch;
                        const float4 a = *reinterpret_cast<const float4*>(stg + ch * 32 + row * 8);
                        const float4 b = *reinterpret_cast<const float4*>(stg + ch * 32 + row * 8 + 4);
                        if (oy + row < direct_win_h<PART>(q) && ox < direct_win_w<PART>(q) && k < q.K) {
                            const float bk = load_bias(q.bias, k);
                            float v[8] = {a.x + bk, a.y + bk, a.z + bk, a.w + bk, b.x + bk, b.y + bk, b.z + bk, b.w + bk};
                            const long long o = (static_cast<long long>(n) * q.K + k) * hw_o + static_cast<long long>(oy + row) * q.Wo + ox;
                            if (q.residual) {
                                const uint4 rv = *reinterpret_cast<const uint4*>(q.residual + o);
                                float f0, f1;
                                unpack2(rv.x, f0, f1); v[0] += f0; v[1] += f1;
                                unpack2(rv.y, f0, f1); v[2] += f0; v[3] += f1;
                                unpack2(rv.z, f0, f1); v[4] += f0; v[5] += f1;
                                unpack2(rv.w, f0, f1); v[6] += f0; v[7] += f1;
                            }
                            if (q.act) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) v[i] = epilogue_act(v[i], q.act);
                            }
                            *reinterpret_cast<uint4*>(q.y + o) =
                                make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
                        }
                    }
                    __syncwarp();
                }
            } else {
                const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(buf * q.n_tile);
                if (q.splits > 1) {
                    float* dst = q.part + static_cast<long long>(wi - work_begin) * q.n_tile * 128 + quarter * 32 + lane;
                    for (int col = half * 16; col < q.n_tile; col += 32) {
                        uint32_t r[16];
                        tmem_ld_32x16_sync(t_addr + col, r);
#pragma unroll
                        for (int j = 0; j < 16; ++j) dst[(col + j) * 128] = __uint_as_float(r[j]);
                    }
                } else {
                    int n, oy, ox;
                    const bool live = direct_out_pixel<PART>(q, m, quarter * 32 + lane, n, oy, ox);
                    const long long yoff = live ? (static_cast<long long>(n) * q.K + k0) * hw_o + static_cast<long long>(oy) * q.Wo + ox : 0;
                    for (int col = half * 16; col < q.n_tile && k0 + col < q.K; col += 32) {
                        uint32_t r[16];
                        tmem_ld_32x16_sync(t_addr + col, r);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            if (live && k0 + col + j < q.K) {
                                float v = __uint_as_float(r[j]) + load_bias(q.bias, k0 + col + j);
                                const long long o = yoff + (col + j) * hw_o;
                                if (q.residual) v += __half2float(q.residual[o]);
                                q.y[o] = __float2half_rn(epilogue_act(v, q.act));
                            }
                        }
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
            buf ^= 1;
            if (buf == 0) acc_phase ^= 1u;
        }
    } else {
        // ------------------------------ patches ------------------------------
        const uint32_t base = smem_u32(a_base), full0 = smem_u32(a_full);
        int as = 0;
        uint32_t aphase = 0;
        bool ok = true;
        pdl_wait();      // the packed copy is the preceding kernel's
        for (int wi = work_begin + blockIdx.x; wi < work_end && ok; wi += gridDim.x) {
            int m, kt, cb0, cb1;
            decode(wi, m, kt, cb0, cb1);
            int row0 = 0, col0 = 0;
            if (!q.flat) {
                // whole images, stride 1: the halo before row and column 0 is filled in by TMA; else it is in the packed copy
                const int org = q.stride == 1 && !PART ? -1 : 0;
                const uint32_t row_blk = fast_div(static_cast<uint32_t>(m), q.fd_tc);
                const uint32_t img = fast_div(row_blk, q.fd_tr);
                col0 = ((m - static_cast<int>(row_blk) * q.tiles_c) * 8 + org) * 8;
                row0 = static_cast<int>(img) * q.rows_img + (static_cast<int>(row_blk) - static_cast<int>(img) * q.tiles_r) * 16 + org;
            }
            for (int cb = cb0; cb < cb1 && ok; ++cb) {
                for (int pl = 0; pl < q.planes; ++pl) {
                    ok = mbar_wait_warp(&a_empty[as], aphase ^ 1u, abort_flag, GEMM_WAIT_LIMIT_NS);
                    if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 7, 0); break; }
                    const uint32_t dst = base + as * q.a_stage_bytes, bar = full0 + as * 8;
                    if (!elected) {
                    } else if (q.flat) {
                        const uint32_t piece = static_cast<uint32_t>(q.PP) * 16u;
                        mbar_arrive_expect_tx_a32(bar, piece * 8u);
                        const __half* src = q.packed + ((static_cast<long long>(pl) * q.pk_pieces + cb * 8) * q.pk_positions +
                                                        static_cast<long long>(m) * 128) * 8;
                        for (int i = 0; i < 8; ++i)
                            bulk_load_a32(dst + i * piece, src + i * q.pk_positions * 8, piece, bar);
                    } else {
                        mbar_arrive_expect_tx_a32(bar, static_cast<uint32_t>(q.PP) * 128u);
                        tma_load_3d_a32(dst, &tmX, bar, col0, row0, pl * q.pk_pieces + cb * 8);
                    }
                    if (++as == q.a_stages) { as = 0; aphase ^= 1u; }
                }
            }
        }
        if (!ok) *abort_flag = 1;
    }
    __syncwarp();
    __syncthreads();
    if (*abort_flag != 0) {
        // copies and MMAs that may still be in flight get a bounded time to land before TMEM and shared memory are released
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

// Adds the fp32 parts of a launch with splits > 1 in a fixed order, then bias, residual, activation, rounding and the
// masked store.  A block of 128 threads = the lanes of one pixel tile; blockIdx.y walks the output channels, two per thread.
template <bool PART>
__global__ void __launch_bounds__(128)
direct_reduce_kernel(const __grid_constant__ DirectParams q, int* __restrict__ status_word) {
    const int pair = q.pair_begin + blockIdx.x;
    const int m = static_cast<int>(fast_div(static_cast<uint32_t>(pair), q.fd_k));
    const int kt = pair - m * q.num_k_tiles;
    const int l = threadIdx.x;
    int n, oy, ox;
    const bool live = direct_out_pixel<PART>(q, m, l, n, oy, ox);
    const long long hw_o = static_cast<long long>(q.Ho) * q.Wo;
    const int col = blockIdx.y * 2, k = kt * q.n_tile + col;
    const long long split_step = static_cast<long long>(q.n_tile) * 128;
    const float* src = q.part + static_cast<long long>(blockIdx.x) * q.splits * split_step + col * 128 + l;
    const long long o = (static_cast<long long>(n) * q.K + k) * hw_o + static_cast<long long>(oy) * q.Wo + ox;
    pdl_launch_dependents();
    pdl_wait();
    if (!wt_header_ok(q.wt_header, q.K, q.C, 1, status_word) || !live || k >= q.K) return;
    float v0 = 0.f, v1 = 0.f;
#pragma unroll 8
    for (int s = 0; s < q.splits; ++s) {
        v0 += __ldcg(src + s * split_step);
        v1 += __ldcg(src + s * split_step + 128);
    }
    v0 += load_bias(q.bias, k);
    if (q.residual) v0 += __half2float(q.residual[o]);
    q.y[o] = __float2half_rn(epilogue_act(v0, q.act));
    if (k + 1 < q.K) {
        v1 += load_bias(q.bias, k + 1);
        if (q.residual) v1 += __half2float(q.residual[o + hw_o]);
        q.y[o + hw_o] = __float2half_rn(epilogue_act(v1, q.act));
    }
}

// x [N][C][H][W] -> [plane][ceil(C / 64) * 8 pieces][positions][8 channels]: the pixels in the order of the flat layout
// (one column and one row of zeros between neighbours, `lead` positions of zeros in front), so that a patch of either
// layout is a few contiguous runs of 16-byte pieces.  Stride 2: plane (a, b) holds pixel (2 r + a - 1, 2 c + b - 1) at
// row r, column c.  A copy of part of the image (see DirectWindow) begins with its halo at row and column -1 of the part, stride
// 1 as well.  One thread per piece: eight 2-byte loads, coalesced over the pixels, one 16-byte store.
__global__ void __launch_bounds__(256)
direct_pack_kernel(const __half* __restrict__ x, uint4* __restrict__ packed, const __grid_constant__ DirectParams q) {
    const long long idx = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    const int piece = blockIdx.y, pl = blockIdx.z;
    const long long Q = idx - q.lead;
    const uint32_t Qu = static_cast<uint32_t>(Q < 0 ? 0 : Q);
    const uint32_t v = fast_div(Qu, q.fd_pkp);
    const uint32_t img = fast_div(v, q.fd_rows);
    const int i = static_cast<int>(v - img * static_cast<uint32_t>(q.rows_img)) * q.stride + (pl >> 1) + q.row0;
    const int j = static_cast<int>(Qu - v * static_cast<uint32_t>(q.pk_pitch)) * q.stride + (pl & 1) + q.col0;
    const bool live = Q >= 0 && static_cast<int>(img) < q.N && static_cast<unsigned>(i) < static_cast<unsigned>(q.H) &&
                      static_cast<unsigned>(j) < static_cast<unsigned>(q.W);
    const long long hw = static_cast<long long>(q.H) * q.W;
    const int c0 = piece * 8;
    const unsigned short* src = reinterpret_cast<const unsigned short*>(x) + (static_cast<long long>(img) * q.C + c0) * hw +
                                static_cast<long long>(i) * q.W + j;
    // wait first, release the convolution second: see the comment on its filters
    pdl_wait();
    pdl_launch_dependents();
    if (idx >= q.pk_positions) return;
    unsigned short h[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) h[c] = live && c0 + c < q.C ? __ldg(src + c * hw) : static_cast<unsigned short>(0);
    packed[(static_cast<long long>(pl) * q.pk_pieces + piece) * q.pk_positions + idx] =
        make_uint4(h[0] | (static_cast<uint32_t>(h[1]) << 16), h[2] | (static_cast<uint32_t>(h[3]) << 16),
                   h[4] | (static_cast<uint32_t>(h[5]) << 16), h[6] | (static_cast<uint32_t>(h[7]) << 16));
}

}  // namespace sdw
