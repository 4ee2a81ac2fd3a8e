// Device code of the folded layout stage (fold.cu has the form and the image's
// layout): used by the split kernels there and by the fused kernel's splitter
// warps.  Included inside an anonymous namespace after tc_ptx.cuh.
#pragma once

constexpr int kFoldRowBytes = kKBlock * 2;          // 64 B per operand row per K block
constexpr int kFoldPart = kTileM * kFoldRowBytes;   // 8 KB: the hi (or lo) parts of a K block

struct FoldSource {
    const float *Q, *U;
    int64_t nlos;               // lines of sight in the cube
    int32_t nchan, nact, chan;  // chan: channel-major
    const int32_t *active;      // [nact]
    const int32_t *padded;      // the same, padded to whole K blocks with a valid channel
};

// L2 eviction priorities of the fused kernel: the cube's data is read once (first out),
// the image ring is rewritten and re-read all the time (last out).
__device__ __forceinline__ uint64_t l2_evict_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_evict_last()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// A load pinned where it stands: as an ordinary read-only load it would be moved down to
// its use, and with it the overlap that the callers arrange.  LAST: the data's last read.
template <bool LAST>
__device__ __forceinline__ float load_here(const float *p)
{
    float v;
    if (LAST) asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(l2_evict_first()));
    else asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// Exponent of a LOS's scale from its largest |value|: the power of two that brings it into
// [2^14, 2^15) (0 for a zero or non-finite one).
__device__ __forceinline__ int fold_exponent(float mx)
{
    int e = 0;
    if (mx > 0.f && isfinite(mx)) {
        frexpf(mx, &e);
        e = 15 - e;
    }
    return max(-100, min(100, e));
}

template <bool RING>
__device__ __forceinline__ void store32(uint8_t *p, const uint32_t (&v)[8], bool swap)
{
    // one 32-byte sector: two 16-byte chunks, exchanged where the swizzle says so
    const uint32_t w[8] = {swap ? v[4] : v[0], swap ? v[5] : v[1], swap ? v[6] : v[2], swap ? v[7] : v[3],
                           swap ? v[0] : v[4], swap ? v[1] : v[5], swap ? v[2] : v[6], swap ? v[3] : v[7]};
    if (RING)
        asm volatile("st.global.L2::cache_hint.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8}, %9;" ::"l"(p), "r"(w[0]), "r"(w[1]),
                     "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "l"(l2_evict_last())
                     : "memory");
    else
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                     "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
}

// 16 channels of one operand row: half hh of the row's 64 bytes in each part.
template <int MODE, bool RING>
__device__ __forceinline__ void emit16(uint8_t *row, int hh, int sw, const float (&v)[16], float scale)
{
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (MODE == MODE_FP16X3) split_pair_fp16(v[2 * j] * scale, v[2 * j + 1] * scale, hi[j], lo[j]);
        else split_pair_bf16(v[2 * j], v[2 * j + 1], hi[j], lo[j]);
    }
    uint8_t *p = row + 32 * (hh ^ (sw >> 1));
    store32<RING>(p, hi, sw & 1);
    if (MODE != MODE_BF16) store32<RING>(p + kFoldPart, lo, sw & 1);
}

// LOS-major rows: a warp takes the 32 active channels of a K block of 8 LOS (one 16-row
// group of a tile).  Lane (half, p) holds channels 2 p and 2 p + 1 of LOS 2 j + half,
// j = 0 .. 3: a load reads two LOS' channels (nearly) contiguously at any alignment,
// flagged channels drop out, and a store writes 64 contiguous bytes of two rows.
// The loads are unconditional, so that all 16 are in flight at once: src_of(r) is row r's
// LOS, or any LOS for a row beyond the end (bit r of dead), whose values become 0 like
// those of padding channels.  v[2 j], v[2 j + 1]: the two channels of LOS 2 j + half.
// Against one channel of 8 LOS per lane, whose 16-bit results were paired by a shuffle and
// stored by every other lane: half the store instructions and no shuffles.  One-kernel form,
// 5,001 LOS x 357 channels x 401 phi BF16x3 37.2 -> 33.2 us, 200,003 LOS FP16x3 0.529 ->
// 0.501 ms, window of 262,144 LOS x 360 -> 64 BF16x3 with its proposal 0.940 -> 0.902 ms.
template <bool LAST, typename F>
__device__ __forceinline__ void fold_load_los(const FoldSource &S, const int *list, int kb, int lane, F src_of, float (&q)[8],
                                              float (&u)[8])
{
    const int2 ch = *reinterpret_cast<const int2 *>(list + kb * kKBlock + 2 * (lane & 15));   // the padded channel list
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int64_t base = src_of(2 * j + (lane >> 4)) * S.nchan;
        q[2 * j] = load_here<LAST>(S.Q + base + ch.x);
        q[2 * j + 1] = load_here<LAST>(S.Q + base + ch.y);
        u[2 * j] = load_here<LAST>(S.U + base + ch.x);
        u[2 * j + 1] = load_here<LAST>(S.U + base + ch.y);
    }
}
__device__ __forceinline__ void fold_mask_los(const FoldSource &S, int kb, int lane, uint32_t dead, float (&q)[8],
                                              float (&u)[8])
{
    const int left = S.nact - kb * kKBlock - 2 * (lane & 15);      // active channels from this lane's first on
    if (__any_sync(0xffffffffu, dead != 0u || left < 2)) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (((dead >> (2 * (e >> 1) + (lane >> 4))) & 1u) || (e & 1) >= left) { q[e] = 0.f; u[e] = 0.f; }
    }
}

// One K block of LOS r0 .. r0 + N - 1 (r0 even) of a group of 8, Q or U; rows: the group's
// first operand row in K block kb of the image; scale[j]: that of LOS r0 + 2 j + half.
template <int MODE, bool RING, int N>
__device__ __forceinline__ void fold_emit_rows(uint8_t *rows, int lane, int r0, const float (&v)[N],
                                               const float (&scale)[N / 2])
{
    const int p = lane & 15, half = lane >> 4;
#pragma unroll
    for (int j = 0; j < N / 2; ++j) {
        const int r = r0 + 2 * j + half;
        uint32_t hi, lo;
        if (MODE == MODE_FP16X3) {
            split_pair_fp16(v[2 * j] * scale[j], v[2 * j + 1] * scale[j], hi, lo);
        } else {
            split_pair_bf16(v[2 * j], v[2 * j + 1], hi, lo);
        }
        uint8_t *at = rows + r * kFoldRowBytes + (((p >> 2) ^ ((r >> 1) & 3)) << 4) + 4 * (p & 3);
        if (RING) {
            asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(at), "r"(hi), "l"(l2_evict_last()) : "memory");
            if (MODE != MODE_BF16)
                asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(at + kFoldPart), "r"(lo), "l"(l2_evict_last()) : "memory");
        } else {
            *reinterpret_cast<uint32_t *>(at) = hi;
            if (MODE != MODE_BF16) *reinterpret_cast<uint32_t *>(at + kFoldPart) = lo;
        }
    }
}
