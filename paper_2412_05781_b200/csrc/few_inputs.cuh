// Layers with few input channels (C <= 4: the 4->320 and 4->512 input convolutions) as one kernel without V, M or a
// workspace.  The contraction is 9 C <= 36 terms long, three steps of the tensor core: for 128 output channels and 128
// consecutive pixels of an image
//   D[k][q] = sum_(tap, c) g[k][(tap, c)] x[(tap, c)][q]
// with the taps g as the A operand and the nine shifted copies of x, gathered pixel by pixel into shared memory, as the B
// operand.  g is taken back out of the transformed filter (see few_outputs.cuh).
//
// A CTA has one block of 128 output channels and every gridDim.x-th tile of 128 pixels.  Warps 0-3 recover the taps and then
// store finished tiles, warps 4-7 gather, warp 8 issues the MMAs.  Lanes of the accumulator are channels: a thread rounds runs
// of pixels of one channel, so they go to shared memory in 16-byte pieces and to y by TMA in whole 128-byte lines.
//
// Bound by the chain of filters, gather, MMA and store, of which two CTAs per SM run side by side: 4->320 at 64x64 (batch 2)
// 7.8 us with fused_small_c_mma_kernel (F(2x2)), 7.3 here, at 128x128 (batch 2) 19.2 -> 11.0, at 96x96 (batch 4) 27.8 -> 11.6,
// 4->512 at 128x128 16.0 -> 9.8.  Relative error (2-norm) against fp64 3.0e-4 instead of 5.2e-4.
#pragma once
#include <cuda_fp16.h>

#include "few_outputs.cuh"
#include "ptx.cuh"
#include "transforms.cuh"

namespace sdw {

constexpr int FI_THREADS = 288;
constexpr int FI_CMAX = 4;
constexpr int FI_K = 128;                      // output channels per CTA (UMMA M)
constexpr int FI_TILE = 128;                   // pixels per tile (UMMA N)
constexpr int FI_STEPS = 3;                    // 9 taps x 4 channels, up to a multiple of 16
constexpr int FI_ROWS_BYTES = 128 * 128;       // 128 rows (channels or pixels) of 64 halves, 48 of them used
constexpr int FI_STG_BYTES = 2 * FI_ROWS_BYTES;            // a finished tile: two boxes [128 k][64 q]
constexpr int FI_SMEM = 3 * FI_ROWS_BYTES + FI_STG_BYTES + 128 + 1024;

struct FewInputsParams {
    const uint32_t* wt_header;
    const __half* U;
    const __half* x;
    const __half* bias;
    int C, K, tile, H, W, hw;
    int Kb;
    int tiles_image, tiles;                    // of 128 pixels: per image, in all
    FastDiv w_div, image_div;
};

// The taps of 128 output channels, row k: (tap, c) -> halves 4 tap + c, 128-byte swizzle; thread k of 128.
template <int M>
__device__ __forceinline__ void fi_recover_taps(const FewInputsParams& q, uint8_t* a_smem, int row, int k) {
    uint2 out[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) out[t] = make_uint2(0, 0);
    if (k < q.K) {
        // rows and columns 0, 1, 2 and the last of U; the first four channels of a row of 64 (zeros past C)
        const uint2* u = reinterpret_cast<const uint2*>(q.U + static_cast<size_t>(k) * 64);
        const size_t plane = static_cast<size_t>(q.Kb) * 1024 / 4;
        uint2 uv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) uv[i][j] = u[((i < 3 ? i : M + 1) * (M + 2) + (j < 3 ? j : M + 1)) * plane];
#pragma unroll
        for (int h = 0; h < 2; ++h) {          // pairs of channels
            float2 t[3][4];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    t[r][j] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float f = fo_left_inverse<M>(r, i);
                        if (f != 0.f) {
                            float a, b;
                            unpack2(h == 0 ? uv[i][j].x : uv[i][j].y, a, b);
                            t[r][j].x = fmaf(f, a, t[r][j].x);
                            t[r][j].y = fmaf(f, b, t[r][j].y);
                        }
                    }
                }
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    float2 g = make_float2(0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float f = fo_left_inverse<M>(s, j);
                        if (f != 0.f) {
                            g.x = fmaf(f, t[r][j].x, g.x);
                            g.y = fmaf(f, t[r][j].y, g.y);
                        }
                    }
                    const __half2 gh = __floats2half2_rn(g.x, g.y);
                    (h == 0 ? out[3 * r + s].x : out[3 * r + s].y) = *reinterpret_cast<const uint32_t*>(&gh);
                }
        }
    }
    uint8_t* dst = a_smem + row * 128;
#pragma unroll
    for (int j = 0; j < 2 * FI_STEPS; ++j) {
        const uint2 lo = 2 * j < 9 ? out[2 * j < 9 ? 2 * j : 0] : make_uint2(0, 0);
        const uint2 hi = 2 * j + 1 < 9 ? out[2 * j + 1 < 9 ? 2 * j + 1 : 0] : make_uint2(0, 0);
        *reinterpret_cast<uint4*>(dst + ((j ^ (row & 7)) << 4)) = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
}

// tmY: fp16 [N][K][H * W], box {64 q, 128 k, 1}, 128-byte swizzle (pixels and channels outside are not written)
__global__ void __launch_bounds__(FI_THREADS, 2)
few_inputs_kernel(const __grid_constant__ CUtensorMap tmY, const FewInputsParams q, int* __restrict__ status_word) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* a_smem = smem;
    uint8_t* b_smem = smem + FI_ROWS_BYTES;                // two tiles
    uint8_t* stg = b_smem + 2 * FI_ROWS_BYTES;
    uint64_t* b_full = reinterpret_cast<uint64_t*>(stg + FI_STG_BYTES);
    uint64_t* b_empty = b_full + 2;
    uint64_t* acc_full = b_empty + 2;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* a_full = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(a_full + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x < 9) {
        // b_full, acc_empty and a_full: one arrival per warp of four; the others: a commit
        mbar_init(&b_full[threadIdx.x], threadIdx.x < 2 || threadIdx.x >= 6 ? 4 : 1);
        fence_barrier_init();
    }
    if (threadIdx.x == 32) {
        *abort_flag = 0;
        prefetch_tmap(&tmY);
    }
    if (warp == 8) { tmem_alloc(tmem_slot, 2 * FI_TILE); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const int k0 = blockIdx.y * FI_K;
    pdl_wait();                 // x and the filters may be the preceding kernel's
    pdl_launch_dependents();
    const bool wt_ok = wt_header_ok(q.wt_header, q.K, q.C, q.tile, status_word);   // the same answer for the whole grid

    if (!wt_ok) {
        // a filter buffer of another layer: nothing is computed
    } else if (warp < 4) {
        // ------------------------------ taps, then y ------------------------------
        const int l = threadIdx.x;             // TMEM lane = output channel
        if (q.tile == 2) fi_recover_taps<2>(q, a_smem, l, k0 + l);
        else fi_recover_taps<4>(q, a_smem, l, k0 + l);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full);
        const float bias = k0 + l < q.K ? load_bias(q.bias, k0 + l) : 0.f;
        int i = 0;
        for (int tile = blockIdx.x; tile < q.tiles; tile += gridDim.x, ++i) {
            const int buf = i & 1;
            if (threadIdx.x == 0) tma_store_wait_read();   // the staging buffer has left
            bool ok = mbar_wait_bounded(&acc_full[buf], (i >> 1) & 1, abort_flag, GEMM_WAIT_LIMIT_NS);
            ok = named_barrier_and(1, 128, ok);            // the four warps give up together or not at all
            if (!ok) {
                if (threadIdx.x == 0) {
                    if (*abort_flag == 0) report_timeout(status_word, 4, 0);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after_sync();
            const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(warp * 32) << 16) + static_cast<uint32_t>(buf * FI_TILE);
#pragma unroll
            for (int c = 0; c < FI_TILE; c += 32) {
                uint32_t r[32];
                tmem_ld_32x32_sync(t_addr + c, r);
                uint8_t* row = stg + (c >> 6) * FI_ROWS_BYTES + l * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t h[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const __half2 v = __floats2half2_rn(__uint_as_float(r[8 * j + 2 * e]) + bias, __uint_as_float(r[8 * j + 2 * e + 1]) + bias);
                        h[e] = *reinterpret_cast<const uint32_t*>(&v);
                    }
                    *reinterpret_cast<uint4*>(row + (((((c & 63) >> 3) + j) ^ (l & 7)) << 4)) = make_uint4(h[0], h[1], h[2], h[3]);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
            fence_proxy_async_smem();
            named_barrier_sync(1, 128);
            if (threadIdx.x == 0) {
                const int img = static_cast<int>(fast_div(static_cast<uint32_t>(tile), q.image_div));
                const int p0 = (tile - img * q.tiles_image) * FI_TILE;
                tma_store_3d(&tmY, stg, p0, k0, img);
                if (p0 + 64 < q.hw) tma_store_3d(&tmY, stg + FI_ROWS_BYTES, p0 + 64, k0, img);
                tma_store_commit();
            }
        }
        if (threadIdx.x == 0) tma_store_wait_all();
    } else if (warp < 8) {
        // ------------------------------ nine shifted copies of x ------------------------------
        const int l = threadIdx.x - 128;       // pixel within the tile
        int i = 0;
        for (int tile = blockIdx.x; tile < q.tiles; tile += gridDim.x, ++i) {
            const int buf = i & 1;
            const int img = static_cast<int>(fast_div(static_cast<uint32_t>(tile), q.image_div));
            const int p = (tile - img * q.tiles_image) * FI_TILE + l;
            const int h = static_cast<int>(fast_div(static_cast<uint32_t>(p), q.w_div)), w = p - h * q.W;
            const unsigned short* src = reinterpret_cast<const unsigned short*>(q.x) + static_cast<long long>(img) * q.C * q.hw + p;
            unsigned short v[9][FI_CMAX];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    const bool in = p < q.hw && static_cast<unsigned>(h + r - 1) < static_cast<unsigned>(q.H) &&
                                    static_cast<unsigned>(w + s - 1) < static_cast<unsigned>(q.W);
#pragma unroll
                    for (int c = 0; c < FI_CMAX; ++c)
                        v[3 * r + s][c] = in && c < q.C ? __ldg(src + static_cast<long long>(c) * q.hw + (r - 1) * q.W + (s - 1))
                                                        : static_cast<unsigned short>(0);
                }
            bool ok = mbar_wait_bounded(&b_empty[buf], ((i >> 1) & 1) ^ 1u, abort_flag, GEMM_WAIT_LIMIT_NS);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) {
                if (lane == 0) {
                    if (*abort_flag == 0) report_timeout(status_word, 1, 0);
                    *abort_flag = 1;
                }
                break;
            }
            uint8_t* dst = b_smem + buf * FI_ROWS_BYTES + l * 128;
            auto two = [&](int t, int c) { return v[t][c] | (static_cast<uint32_t>(v[t][c + 1]) << 16); };
#pragma unroll
            for (int j = 0; j < 2 * FI_STEPS; ++j) {
                uint4 piece = make_uint4(0, 0, 0, 0);
                if (2 * j < 9) { piece.x = two(2 * j < 9 ? 2 * j : 0, 0); piece.y = two(2 * j < 9 ? 2 * j : 0, 2); }
                if (2 * j + 1 < 9) { piece.z = two(2 * j + 1 < 9 ? 2 * j + 1 : 0, 0); piece.w = two(2 * j + 1 < 9 ? 2 * j + 1 : 0, 2); }
                *reinterpret_cast<uint4*>(dst + ((j ^ (l & 7)) << 4)) = piece;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&b_full[buf]);
        }
    } else {
        // ------------------------------ MMA ------------------------------
        const bool elected = elect_one() != 0;
        const uint32_t idesc = make_idesc_f16_f32(FI_K, FI_TILE, false, false);
        const uint64_t adesc = make_smem_desc_sw128(smem_u32(a_smem), 16, 1024);
        const uint64_t bdesc0 = make_smem_desc_sw128(smem_u32(b_smem), 16, 1024);
        bool ok = mbar_wait_warp(a_full, 0u, abort_flag, GEMM_WAIT_LIMIT_NS);
        if (!ok && *abort_flag == 0) report_timeout(status_word, 6, 0);
        int i = 0;
        for (int tile = blockIdx.x; tile < q.tiles && ok; tile += gridDim.x, ++i) {
            const int buf = i & 1;
            ok = mbar_wait_warp(&acc_empty[buf], ((i >> 1) & 1) ^ 1u, abort_flag, GEMM_WAIT_LIMIT_NS);
            if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 2, 0); break; }
            ok = mbar_wait_warp(&b_full[buf], (i >> 1) & 1, abort_flag, GEMM_WAIT_LIMIT_NS);
            if (!ok) { if (*abort_flag == 0) report_timeout(status_word, 3, 0); break; }
            tc_fence_after_sync();
            if (elected) {
                const uint64_t bdesc = bdesc0 + static_cast<uint64_t>(buf * (FI_ROWS_BYTES >> 4));
#pragma unroll
                for (int s = 0; s < FI_STEPS; ++s)
                    umma_f16(tmem_base + static_cast<uint32_t>(buf * FI_TILE), adesc + 2 * s, bdesc + 2 * s, idesc, s > 0 ? 1u : 0u);
                umma_commit(&b_empty[buf]);
                umma_commit(&acc_full[buf]);
            }
        }
        if (!ok) *abort_flag = 1;
    }

    __syncwarp();
    __syncthreads();
    if (*abort_flag != 0) {
        // copies and MMAs that may still be in flight get a bounded time to land before their memory is released
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 8) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 2 * FI_TILE);
    }
}

}  // namespace sdw
