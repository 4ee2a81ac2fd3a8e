// Layout stage of folded grids: FP32 Q/U -> the 16-bit operand image of the
// folded contraction.
//
// On a phi grid symmetric about zero, cos(2 phi x) is even and sin(2 phi x) odd
// in phi, so with the four sums over channels
//     Qc = sum Q c,  Qs = sum Q s,  Uc = sum U c,  Us = sum U s      (phi >= 0)
// Eq. Fsum gives both
//     F(+phi) = (Qc + Us) + i (Uc - Qs)   and   F(-phi) = (Qc - Us) + i (Uc + Qs):
// four real multiply-adds per (channel, pair of depths) where evaluating each
// depth by itself takes eight.  As a matrix product that is [Q; U] [c | s], with
// Q and U as rows of their own (K = channels), half the phase columns and half
// the K of the interleaved form.
//
// Image: per tile of 64 LOS and K block of 32 active channels, 128 rows x 64
// bytes of hi parts, then of lo parts.  LOS i of the tile has its Q in row
// 16 (i / 8) + i % 8 and its U eight rows below, so that the contraction's
// 16-lane TMEM loads hand one thread Qc, Qs, Uc, Us of a LOS.  Rows are swizzled
// as the MMA reads them: 16-byte chunk c of row r at r * 64 + ((c ^ ((r >> 1) & 3)) << 4).
//
// Measured against the interleaved form (whole call, BF16x3 unless stated; GB300):
//   262,144 LOS x 360 active channels x 401 phi   0.931 -> 0.663 ms
//   160,000 x 1536 x 4001                         15.4  -> 7.76 ms
//   200,000 x 856 x 7000, peak map only           18.6  -> 8.17 ms
//   400,000 x 800 x 1001, plain BF16              2.99  -> 2.12 ms
//
// Both kernels are bound by HBM: 8 bytes read and 8 written per (LOS, active channel),
// 0.255 ms for the first cube (5.9 TB/s of the measured 6.8 copy bandwidth).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "rms_internal.h"

namespace {

#include "tc_ptx.cuh"
#include "fold_split.cuh"

constexpr int kLosPerCta = 2 * kFoldTileLos;
constexpr int kBlock = 2 * kFoldPart;           // image bytes per K block of a tile: hi then lo parts

struct FoldSplitParams {
    FoldSource src;
    const int64_t *rows;        // optional gather: image LOS i <- cube LOS rows[i]
    const int64_t *count;       // optional device count of image LOS: tiles past it stay untouched
    int32_t kblocks;
    int32_t kpg;                // K blocks per CTA: blockIdx.y covers K blocks [y kpg, (y + 1) kpg)
    uint8_t *A;                 // [ceil(nlos / 128) 2][kblocks][16 KB]
    int8_t *rexp;               // [nlos] (FP16X3): the LOS's exponent
};

// Channel-major cubes: one thread per LOS, 128 LOS (two tiles) per CTA; a warp
// reads 128 contiguous bytes of a channel row.
template <int MODE>
__global__ void __launch_bounds__(kLosPerCta) fold_split_chan_kernel(const FoldSplitParams P)
{
    const int m = threadIdx.x;
    const int64_t n = P.count ? min(*P.count, P.src.nlos) : P.src.nlos;
    if ((int64_t)blockIdx.x * kLosPerCta >= n) return;
    const int64_t los = (int64_t)blockIdx.x * kLosPerCta + m;
    const bool valid = los < n;
    const int64_t src = P.rows && valid ? P.rows[los] : los;
    const int i = m & (kFoldTileLos - 1), r = 16 * (i >> 3) + (i & 7), sw = (r >> 1) & 3;
    const int kb0 = (int)blockIdx.y * P.kpg, kb1 = min(P.kblocks, kb0 + P.kpg);
    uint8_t *const tile = P.A + ((size_t)blockIdx.x * 2 + (m / kFoldTileLos)) * P.kblocks * kBlock + r * kFoldRowBytes;
    auto load = [&](int c0, float (&q)[16], float (&u)[16]) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            q[j] = 0.f;
            u[j] = 0.f;
            if (c0 + j < P.src.nact && valid) {
                const int64_t off = (int64_t)__ldg(P.src.active + c0 + j) * P.src.nlos + src;
                q[j] = __ldg(P.src.Q + off);
                u[j] = __ldg(P.src.U + off);
            }
        }
    };
    float scale = 1.0f;
    if (MODE == MODE_FP16X3) {
        float mx = 0.f;
        for (int c0 = 0; c0 < P.src.nact; c0 += 16) {
            float q[16], u[16];
            load(c0, q, u);
#pragma unroll
            for (int j = 0; j < 16; ++j) mx = fmaxf(mx, fmaxf(fabsf(q[j]), fabsf(u[j])));
        }
        const int e = fold_exponent(mx);
        scale = ldexpf(1.0f, e);
        if (valid) P.rexp[los] = (int8_t)e;
    }
    for (int h = 2 * kb0; h < 2 * kb1; ++h) {
        float q[16], u[16];
        load(16 * h, q, u);
        uint8_t *row = tile + (size_t)(h >> 1) * kBlock;
        emit16<MODE, false>(row, h & 1, sw, q, scale);
        emit16<MODE, false>(row + 8 * kFoldRowBytes, h & 1, sw, u, scale);
    }
}

// LOS-major cubes: one tile of 64 LOS per CTA, 8 LOS per warp.
template <int MODE>
__global__ void __launch_bounds__(256, MODE == MODE_FP16X3 ? 3 : 4) fold_split_los_kernel(const FoldSplitParams P)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = P.count ? min(*P.count, P.src.nlos) : P.src.nlos;
    if ((int64_t)blockIdx.x * kFoldTileLos >= n) return;
    const int64_t los0 = ((int64_t)blockIdx.x * 8 + warp) * 8;
    const int kb0 = (int)blockIdx.y * P.kpg, kb1 = min(P.kblocks, kb0 + P.kpg);
    uint8_t *const group = P.A + (size_t)blockIdx.x * P.kblocks * kBlock + 16 * warp * kFoldRowBytes;
    auto src_of = [&](int r) -> int64_t {
        const int64_t los = min(los0 + r, n - 1);
        return P.rows ? __ldg(P.rows + los) : los;
    };
    const uint32_t dead = los0 + 8 <= n ? 0u : (0xffu << max(0, (int)(n - los0))) & 0xffu;
    float scale[8];
    if constexpr (MODE == MODE_FP16X3) {
        int ex[8];
        fold_scales_los(P.src, P.src.padded, P.kblocks, lane, src_of, dead, scale, ex);
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (lane == r && los0 + r < n) P.rexp[los0 + r] = (int8_t)ex[r];
    }
    for (int kb = kb0; kb < kb1; ++kb) {
        float q[8], u[8];
        fold_load_los<false>(P.src, P.src.padded, kb, lane, src_of, q, u);
        fold_mask_los(P.src, kb, lane, dead, q, u);
        fold_emit_rows<MODE, false, 8>(group + (size_t)kb * kBlock, lane, 0, q, scale);
        fold_emit_rows<MODE, false, 8>(group + (size_t)kb * kBlock + 8 * kFoldRowBytes, lane, 0, u, scale);
    }
}

}  // namespace

cudaError_t launch_fold_split(const rms_plan_s &p, const float *Q, const float *U, int64_t nlos, int layout,
                              uint8_t *A, int8_t *rexp, cudaStream_t s, const int64_t *rows, const int64_t *count)
{
    const int mode = mode_of(p.precision);
    const bool chan = layout == RMS_CHAN_MAJOR;
    // the image has an even number of 64-LOS tiles: a padding tile is written as zeros
    const int64_t pairs = (nlos + kLosPerCta - 1) / kLosPerCta;
    const int64_t nb = chan ? pairs : 2 * pairs;
    if (nb < 1) return cudaSuccess;
    if (nb > 0x7fffffff) return cudaErrorInvalidValue;
    if (mode == MODE_FP16X3 && !rexp) return cudaErrorInvalidValue;
    FoldSplitParams P;
    P.src = {Q, U, nlos, p.nchan, p.nact, chan, p.d_active, p.fold.d_list};
    P.rows = rows;
    P.count = count;
    P.kblocks = p.fold.kblocks;
    P.A = A;
    P.rexp = rexp;
    // K blocks of a tile are shared out over blockIdx.y until the grid is about 8 waves
    // (8-9 CTAs of 128 threads per SM, 4 of 256); FP16X3 needs a LOS's whole row
    int64_t groups = 1;
    if (mode != MODE_FP16X3) {
        const int64_t target = (int64_t)8 * (chan ? 9 : 4) * p.num_sms;
        groups = std::min<int64_t>(P.kblocks, std::max<int64_t>(1, (target + nb - 1) / nb));
    }
    P.kpg = (int32_t)((P.kblocks + groups - 1) / groups);
    const dim3 grid((unsigned)nb, (unsigned)((P.kblocks + P.kpg - 1) / P.kpg));
    if (chan) {
        if (mode == MODE_BF16) fold_split_chan_kernel<MODE_BF16><<<grid, kLosPerCta, 0, s>>>(P);
        else if (mode == MODE_BF16X3) fold_split_chan_kernel<MODE_BF16X3><<<grid, kLosPerCta, 0, s>>>(P);
        else fold_split_chan_kernel<MODE_FP16X3><<<grid, kLosPerCta, 0, s>>>(P);
    } else {
        if (mode == MODE_BF16) fold_split_los_kernel<MODE_BF16><<<grid, 256, 0, s>>>(P);
        else if (mode == MODE_BF16X3) fold_split_los_kernel<MODE_BF16X3><<<grid, 256, 0, s>>>(P);
        else fold_split_los_kernel<MODE_FP16X3><<<grid, 256, 0, s>>>(P);
    }
    return cudaGetLastError();
}
