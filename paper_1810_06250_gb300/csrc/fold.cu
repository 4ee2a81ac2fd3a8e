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
    const int8_t *rexp;         // [nlos] (FP16X3): the LOS's exponent
};

// FP16X3: the exponent of every LOS's scale, from its largest active |value|, in a pass of its
// own at copy bandwidth, so that what follows (the split, or the one-kernel form) can take a
// LOS's channels in any order and by any number of CTAs.  It took the place of passes inside
// the split (one thread walked a LOS's channels twice) and inside the one-kernel form (whose
// warps waited for each other's maxima, LOS-major only).  Whole call, channel-major:
// 262,144 LOS x 360 x 401 0.808 -> 0.597 ms, 60,000 x 1350 x 301 0.804 -> 0.544, 8,506 x 416 x
// 497 121 -> 56 us, 3,000 x 360 x 401 96 -> 43 us; LOS-major 0.631 -> 0.610, 0.623 -> 0.555 ms,
// 54 -> 54, 48 -> 45 us.
// Channel-major: 128 LOS per CTA, four per lane, the channels dealt out to 16 warps; VEC:
// rows start on 16 bytes.  0.127 ms for the first cube: 5.9 TB/s.
constexpr int kExpWarps = 16, kExpBatch = 8;
template <bool VEC>
__global__ void __launch_bounds__(32 * kExpWarps) fold_exp_chan_kernel(const FoldSource S, int8_t *rexp)
{
    __shared__ float part[kExpWarps][kLosPerCta];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t los0 = (int64_t)blockIdx.x * kLosPerCta;
    auto at = [&](int k) { return min(los0 + lane + 32 * k, S.nlos - 1); };          // beyond the end: any LOS
    const int64_t at4 = min(los0 + 4 * lane, S.nlos - 4);
    float mx[4] = {0.f, 0.f, 0.f, 0.f};
    // the warp's channels warp, warp + 16, ..: their numbers first, one per lane, so that all of a
    // batch's loads are in flight at once (a number beyond the last is the last channel's again)
    for (int a0 = warp; a0 < S.nact; a0 += 32 * kExpWarps) {
        const int mine = __ldg(S.active + min(a0 + kExpWarps * lane, S.nact - 1));
        const int nj = min(32, (S.nact - a0 + kExpWarps - 1) / kExpWarps);
        for (int j0 = 0; j0 < nj; j0 += kExpBatch) {
            float q[kExpBatch][4], u[kExpBatch][4];
#pragma unroll
            for (int j = 0; j < kExpBatch; ++j) {
                const int64_t row = (int64_t)__shfl_sync(0xffffffffu, mine, j0 + j) * S.nlos;
                if (VEC) {
                    const float4 x = __ldg(reinterpret_cast<const float4 *>(S.Q + row + at4));
                    const float4 y = __ldg(reinterpret_cast<const float4 *>(S.U + row + at4));
                    q[j][0] = x.x; q[j][1] = x.y; q[j][2] = x.z; q[j][3] = x.w;
                    u[j][0] = y.x; u[j][1] = y.y; u[j][2] = y.z; u[j][3] = y.w;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        q[j][k] = __ldg(S.Q + row + at(k));
                        u[j][k] = __ldg(S.U + row + at(k));
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < kExpBatch; ++j)
#pragma unroll
                for (int k = 0; k < 4; ++k) mx[k] = fmaxf(mx[k], fmaxf(fabsf(q[j][k]), fabsf(u[j][k])));
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) part[warp][VEC ? 4 * lane + k : lane + 32 * k] = mx[k];
    __syncthreads();
    const int64_t los = los0 + threadIdx.x;
    if (threadIdx.x < kLosPerCta && los < S.nlos) {
        float m = part[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < kExpWarps; ++w) m = fmaxf(m, part[w][threadIdx.x]);
        rexp[los] = (int8_t)fold_exponent(m);
    }
}

// LOS-major: a warp per LOS (the list's padding repeats an active channel).
__global__ void __launch_bounds__(256) fold_exp_los_kernel(const FoldSource S, int32_t kblocks, int8_t *rexp)
{
    const int lane = threadIdx.x & 31;
    const int64_t los = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (los >= S.nlos) return;
    const float *q = S.Q + los * S.nchan, *u = S.U + los * S.nchan;
    float mx = 0.f;
#pragma unroll 4
    for (int kb = 0; kb < kblocks; ++kb) {
        const int c = __ldg(S.padded + kb * kKBlock + lane);
        mx = fmaxf(mx, fmaxf(fabsf(__ldg(q + c)), fabsf(__ldg(u + c))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) rexp[los] = (int8_t)fold_exponent(mx);
}

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
    const float scale = MODE == MODE_FP16X3 ? ldexpf(1.0f, __ldg(P.rexp + min(los, n - 1))) : 1.0f;
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
__global__ void __launch_bounds__(256, 4) fold_split_los_kernel(const FoldSplitParams P)
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
    float scale[4];
    if constexpr (MODE == MODE_FP16X3) {
#pragma unroll
        for (int j = 0; j < 4; ++j) scale[j] = ldexpf(1.0f, __ldg(P.rexp + min(los0 + 2 * j + (lane >> 4), n - 1)));
    }
    for (int kb = kb0; kb < kb1; ++kb) {
        float q[8], u[8];
        fold_load_los<false>(P.src, P.src.padded, kb, lane, src_of, q, u);
        fold_mask_los(P.src, kb, lane, dead, q, u);
        fold_emit_rows<MODE, false, 8>(group + (size_t)kb * kBlock, lane, 0, q, scale);
        fold_emit_rows<MODE, false, 8>(group + (size_t)kb * kBlock + 8 * kFoldRowBytes, lane, 0, u, scale);
    }
}

// The folded image of gathered lines of sight, from an interleaved image (gemm.cu) that holds the same 16-bit parts: one
// 64-LOS tile and K block per CTA, 8 channels of a LOS per thread.  A row's 64 bytes per 16 channels are contiguous there,
// where a channel-major cube gives one value of every 32-byte sector to a gathered LOS.
__global__ void __launch_bounds__(4 * kFoldTileLos) fold_gather_kernel(const uint8_t *src, int32_t src_kblocks,
                                                                       const int32_t *column, int32_t nact,
                                                                       const int64_t *rows, const int64_t *count,
                                                                       int64_t nmax, int32_t parts, uint8_t *dst)
{
    const int i = threadIdx.x >> 2, c = threadIdx.x & 3, kb = blockIdx.y;
    const int64_t n = min(*count, nmax), j = (int64_t)blockIdx.x * kFoldTileLos + i;
    if ((int64_t)blockIdx.x * kFoldTileLos >= n) return;
    const int64_t r = rows[min(j, n - 1)];
    const int ms = (int)(r % kTileM), sws = (ms >> 1) & 3;
    const uint8_t *const from = src + (size_t)(r / kTileM) * src_kblocks * kBlock + ms * kFoldRowBytes;
    const int at = 16 * (i >> 3) + (i & 7), sw = (at >> 1) & 3;
    uint8_t *const to = dst + ((size_t)blockIdx.x * gridDim.y + kb) * kBlock + at * kFoldRowBytes + ((c ^ sw) << 4);
    for (int part = 0; part < parts; ++part) {
        uint32_t v[8];                  // (Q, U) of 8 channels
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int a = kb * kKBlock + 8 * c + e;
            v[e] = 0u;
            if (a < nact && j < n) {
                const int ch = column ? __ldg(column + a) : a;
                v[e] = *reinterpret_cast<const uint32_t *>(from + (size_t)(ch >> 4) * kBlock + part * kFoldPart +
                                                           ((((ch >> 2) & 3) ^ sws) << 4) + 4 * (ch & 3));
            }
        }
        uint32_t q[4], u[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            q[e] = __byte_perm(v[2 * e], v[2 * e + 1], 0x5410);
            u[e] = __byte_perm(v[2 * e], v[2 * e + 1], 0x7632);
        }
        *reinterpret_cast<uint4 *>(to + part * kFoldPart) = make_uint4(q[0], q[1], q[2], q[3]);
        *reinterpret_cast<uint4 *>(to + part * kFoldPart + 8 * kFoldRowBytes) = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

}  // namespace

cudaError_t launch_fold_gather(const rms_plan_s &p, int layout, const uint8_t *src, const int64_t *rows,
                               const int64_t *count, int64_t nmax, uint8_t *dst, cudaStream_t s)
{
    const bool chan = layout == RMS_CHAN_MAJOR;
    const int64_t tiles = (nmax + kFoldTileLos - 1) / kFoldTileLos;
    if (tiles < 1) return cudaSuccess;
    if (tiles > 0x7fffffff || p.fold.kblocks > 65535) return cudaErrorInvalidValue;
    // a channel-major image's columns are the active channels, a LOS-major one's all channels
    fold_gather_kernel<<<dim3((unsigned)tiles, (unsigned)p.fold.kblocks), 4 * kFoldTileLos, 0, s>>>(
        src, chan ? p.kblocks : p.kblocks_raw, chan ? nullptr : p.d_active, p.nact, rows, count, nmax,
        p.precision == RMS_BF16 ? 1 : 2, dst);
    return cudaGetLastError();
}

cudaError_t launch_fold_exponents(const rms_plan_s &p, const float *Q, const float *U, int64_t nlos, int layout,
                                  int8_t *rexp, cudaStream_t s)
{
    const bool chan = layout == RMS_CHAN_MAJOR;
    const FoldSource src = {Q, U, nlos, p.nchan, p.nact, chan, p.d_active, p.fold.d_list};
    const int64_t nb = chan ? (nlos + kLosPerCta - 1) / kLosPerCta : (nlos + 7) / 8;
    if (nb < 1) return cudaSuccess;
    if (nb > 0x7fffffff) return cudaErrorInvalidValue;
    const bool vec = nlos % 4 == 0 && !((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(U)) & 15);
    if (!chan) fold_exp_los_kernel<<<(unsigned)nb, 256, 0, s>>>(src, p.fold.kblocks, rexp);
    else if (vec) fold_exp_chan_kernel<true><<<(unsigned)nb, 32 * kExpWarps, 0, s>>>(src, rexp);
    else fold_exp_chan_kernel<false><<<(unsigned)nb, 32 * kExpWarps, 0, s>>>(src, rexp);
    return cudaGetLastError();
}

cudaError_t launch_fold_split(const rms_plan_s &p, const float *Q, const float *U, int64_t nlos, int layout,
                              uint8_t *A, int8_t *rexp, cudaStream_t s, const int64_t *rows, const int64_t *count)
{
    const int mode = mode_of(p.precision);
    const bool chan = layout == RMS_CHAN_MAJOR;
    // the image has an even number of 64-LOS tiles: a padding tile is zeros channel-major, and stays
    // unwritten LOS-major (its rows reach no output, and no other row)
    const int64_t pairs = (nlos + kLosPerCta - 1) / kLosPerCta;
    const int64_t nb = chan ? pairs : 2 * pairs;
    if (nb < 1) return cudaSuccess;
    if (nb > 0x7fffffff) return cudaErrorInvalidValue;
    if (mode == MODE_FP16X3) {
        if (!rexp || rows || count) return cudaErrorInvalidValue;      // (only BF16 plans gather)
        const cudaError_t e = launch_fold_exponents(p, Q, U, nlos, layout, rexp, s);
        if (e != cudaSuccess) return e;
    }
    FoldSplitParams P;
    P.src = {Q, U, nlos, p.nchan, p.nact, chan, p.d_active, p.fold.d_list};
    P.rows = rows;
    P.count = count;
    P.kblocks = p.fold.kblocks;
    P.A = A;
    P.rexp = rexp;
    // K blocks of a tile are shared out over blockIdx.y until the grid is about 8 waves
    // (8-9 CTAs of 128 threads per SM, 4 of 256)
    const int64_t target = (int64_t)8 * (chan ? 9 : 4) * p.num_sms;
    const int64_t groups = std::min<int64_t>(P.kblocks, std::max<int64_t>(1, (target + nb - 1) / nb));
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
