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

constexpr int kRowBytes = kKBlock * 2;          // 64 B per operand row per K block
constexpr int kPart = kTileM * kRowBytes;       // 8 KB: the hi (or lo) parts of a K block
constexpr int kLosPerCta = 2 * kFoldTileLos;

struct FoldSplitParams {
    const float *Q, *U;
    int64_t nlos;               // lines of sight in the cube
    const int64_t *rows;        // optional gather: image LOS i <- cube LOS rows[i]
    const int64_t *count;       // optional device count of image LOS: tiles past it stay untouched
    int32_t nchan, nact, kblocks;
    int32_t kpg;                // K blocks per CTA: blockIdx.y covers K blocks [y kpg, (y + 1) kpg)
    const int32_t *active;
    uint8_t *A;                 // [ceil(nlos / 128) 2][kblocks][16 KB]
    int8_t *rexp;               // [nlos] (FP16X3): power of two that brings the LOS's largest |value| into [2^14, 2^15)
};

// Exponent of a LOS's scale from its largest |value| (0 for a zero or non-finite one).
__device__ __forceinline__ int row_exponent(float mx)
{
    int e = 0;
    if (mx > 0.f && isfinite(mx)) {
        frexpf(mx, &e);
        e = 15 - e;
    }
    return max(-100, min(100, e));
}

__device__ __forceinline__ void store32(uint8_t *p, const uint32_t (&v)[8], bool swap)
{
    // one 32-byte sector: two 16-byte chunks, exchanged where the swizzle says so
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(swap ? v[4] : v[0]),
                 "r"(swap ? v[5] : v[1]), "r"(swap ? v[6] : v[2]), "r"(swap ? v[7] : v[3]), "r"(swap ? v[0] : v[4]),
                 "r"(swap ? v[1] : v[5]), "r"(swap ? v[2] : v[6]), "r"(swap ? v[3] : v[7])
                 : "memory");
}

// 16 channels of one operand row: half hh of the row's 64 bytes in each part.
template <int MODE>
__device__ __forceinline__ void emit16(uint8_t *row, int hh, int sw, const float (&v)[16], float scale)
{
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (MODE == MODE_FP16X3) split_pair_fp16(v[2 * j] * scale, v[2 * j + 1] * scale, hi[j], lo[j]);
        else split_pair_bf16(v[2 * j], v[2 * j + 1], hi[j], lo[j]);
    }
    uint8_t *p = row + 32 * (hh ^ (sw >> 1));
    store32(p, hi, sw & 1);
    if (MODE != MODE_BF16) store32(p + kPart, lo, sw & 1);
}

// Channel-major cubes: one thread per LOS, 128 LOS (two tiles) per CTA; a warp
// reads 128 contiguous bytes of a channel row.
template <int MODE>
__global__ void __launch_bounds__(kLosPerCta) fold_split_chan_kernel(const FoldSplitParams P)
{
    const int m = threadIdx.x;
    const int64_t n = P.count ? min(*P.count, P.nlos) : P.nlos;
    if ((int64_t)blockIdx.x * kLosPerCta >= n) return;
    const int64_t los = (int64_t)blockIdx.x * kLosPerCta + m;
    const bool valid = los < n;
    const int64_t src = P.rows && valid ? P.rows[los] : los;
    const int i = m & (kFoldTileLos - 1), r = 16 * (i >> 3) + (i & 7), sw = (r >> 1) & 3;
    const int kb0 = (int)blockIdx.y * P.kpg, kb1 = min(P.kblocks, kb0 + P.kpg);
    uint8_t *const tile = P.A + ((size_t)blockIdx.x * 2 + (m / kFoldTileLos)) * P.kblocks * (2 * kPart) + r * kRowBytes;
    auto load = [&](int c0, float (&q)[16], float (&u)[16]) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            q[j] = 0.f;
            u[j] = 0.f;
            if (c0 + j < P.nact && valid) {
                const int64_t off = (int64_t)__ldg(P.active + c0 + j) * P.nlos + src;
                q[j] = __ldg(P.Q + off);
                u[j] = __ldg(P.U + off);
            }
        }
    };
    float scale = 1.0f;
    if (MODE == MODE_FP16X3) {
        float mx = 0.f;
        for (int c0 = 0; c0 < P.nact; c0 += 16) {
            float q[16], u[16];
            load(c0, q, u);
#pragma unroll
            for (int j = 0; j < 16; ++j) mx = fmaxf(mx, fmaxf(fabsf(q[j]), fabsf(u[j])));
        }
        const int e = row_exponent(mx);
        scale = ldexpf(1.0f, e);
        if (valid) P.rexp[los] = (int8_t)e;
    }
    for (int h = 2 * kb0; h < 2 * kb1; ++h) {
        float q[16], u[16];
        load(16 * h, q, u);
        uint8_t *row = tile + (size_t)(h >> 1) * (2 * kPart);
        emit16<MODE>(row, h & 1, sw, q, scale);
        emit16<MODE>(row + 8 * kRowBytes, h & 1, sw, u, scale);
    }
}

// hi and lo 16-bit parts of one value, hi in the low half.
template <int MODE>
__device__ __forceinline__ uint32_t split_one(float v)
{
    if (MODE == MODE_FP16X3) {
        const __half h = __float2half_rn(v);
        const __half l = __float2half_rn(v - __half2float(h));
        return (uint32_t)__half_as_ushort(h) | ((uint32_t)__half_as_ushort(l) << 16);
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const __nv_bfloat16 l = __float2bfloat16_rn(v - __bfloat162float(h));
    return (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(l) << 16);
}

// LOS-major cubes: a warp takes 8 LOS (one 16-row group of a tile) and its lanes
// the 32 active channels of a K block, so that a load reads a LOS's channels
// (nearly) contiguously at any alignment, flagged channels drop out, and after an
// exchange between lane pairs (even lanes take the hi words, odd lanes the lo
// words) a store writes 64 contiguous bytes of each part.
template <int MODE>
__global__ void __launch_bounds__(256) fold_split_los_kernel(const FoldSplitParams P)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = P.count ? min(*P.count, P.nlos) : P.nlos;
    if ((int64_t)blockIdx.x * kFoldTileLos >= n) return;
    const int64_t los0 = ((int64_t)blockIdx.x * 8 + warp) * 8;     // 64 LOS, one tile, per CTA
    const int kb0 = (int)blockIdx.y * P.kpg, kb1 = min(P.kblocks, kb0 + P.kpg);
    uint8_t *const group = P.A + (size_t)blockIdx.x * P.kblocks * (2 * kPart) + 16 * warp * kRowBytes +
                           ((lane & 1) ? kPart : 0) + 4 * ((lane >> 1) & 3);
    const int chunk = lane >> 3;
    auto load = [&](int kb, float (&q)[8], float (&u)[8]) {
        const int c = kb * kKBlock + lane;
        const int ch = c < P.nact ? __ldg(P.active + c) : -1;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            q[r] = 0.f;
            u[r] = 0.f;
            if (ch >= 0 && los0 + r < n) {
                const int64_t off = (P.rows ? __ldg(P.rows + los0 + r) : los0 + r) * P.nchan + ch;
                q[r] = __ldg(P.Q + off);
                u[r] = __ldg(P.U + off);
            }
        }
    };
    float scale[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) scale[r] = 1.0f;
    if (MODE == MODE_FP16X3) {
        float mx[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) mx[r] = 0.f;
        for (int kb = 0; kb < P.kblocks; ++kb) {
            float q[8], u[8];
            load(kb, q, u);
#pragma unroll
            for (int r = 0; r < 8; ++r) mx[r] = fmaxf(mx[r], fmaxf(fabsf(q[r]), fabsf(u[r])));
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], o));
            const int e = row_exponent(mx[r]);
            scale[r] = ldexpf(1.0f, e);
            if (lane == r && los0 + r < n) P.rexp[los0 + r] = (int8_t)e;
        }
    }
    for (int kb = kb0; kb < kb1; ++kb) {
        float q[8], u[8];
        load(kb, q, u);
        uint8_t *blk = group + (size_t)kb * (2 * kPart);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint32_t wq = split_one<MODE>(MODE == MODE_FP16X3 ? q[r] * scale[r] : q[r]);
            const uint32_t wu = split_one<MODE>(MODE == MODE_FP16X3 ? u[r] * scale[r] : u[r]);
            const uint32_t pq = __shfl_xor_sync(0xffffffffu, wq, 1), pu = __shfl_xor_sync(0xffffffffu, wu, 1);
            const uint32_t oq = (lane & 1) ? __byte_perm(pq, wq, 0x7632) : __byte_perm(wq, pq, 0x5410);
            const uint32_t ou = (lane & 1) ? __byte_perm(pu, wu, 0x7632) : __byte_perm(wu, pu, 0x5410);
            uint8_t *p = blk + r * kRowBytes + ((chunk ^ ((r >> 1) & 3)) << 4);
            if (MODE != MODE_BF16 || !(lane & 1)) {
                *reinterpret_cast<uint32_t *>(p) = oq;
                *reinterpret_cast<uint32_t *>(p + 8 * kRowBytes) = ou;
            }
        }
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
    P.Q = Q;
    P.U = U;
    P.nlos = nlos;
    P.rows = rows;
    P.count = count;
    P.nchan = p.nchan;
    P.nact = p.nact;
    P.kblocks = p.fold.kblocks;
    P.active = p.d_active;
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
