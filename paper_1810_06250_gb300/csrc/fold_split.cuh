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

// LOS-major rows: the lanes of a warp take the 32 active channels of a K block of 8 LOS
// (one 16-row group of a tile), so that a load reads a LOS's channels (nearly)
// contiguously at any alignment, flagged channels drop out, and after an exchange
// between lane pairs (even lanes take the hi words, odd lanes the lo words) a store
// writes 64 contiguous bytes of each part.  The loads are unconditional, so that all 16
// are in flight at once: src_of(r) is row r's LOS, or any LOS for a row beyond the end
// (bit r of dead), whose values become 0 like those of padding channels.
template <bool LAST, typename F>
__device__ __forceinline__ void fold_load_los(const FoldSource &S, const int *list, int kb, int lane, F src_of, float (&q)[8],
                                              float (&u)[8])
{
    const int ch = list[kb * kKBlock + lane];      // the padded channel list
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int64_t off = src_of(r) * S.nchan + ch;
        q[r] = load_here<LAST>(S.Q + off);
        u[r] = load_here<LAST>(S.U + off);
    }
}
__device__ __forceinline__ void fold_mask_los(const FoldSource &S, int kb, int lane, uint32_t dead, float (&q)[8],
                                              float (&u)[8])
{
    if (kb * kKBlock + lane >= S.nact) dead = 0xffu;
    if (__any_sync(0xffffffffu, dead != 0u)) {
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if ((dead >> r) & 1u) { q[r] = 0.f; u[r] = 0.f; }
    }
}

// The scales (and exponents) of 8 LOS: a first pass over their rows.
template <typename F>
__device__ __forceinline__ void fold_scales_los(const FoldSource &S, const int *list, int kblocks, int lane, F src_of, uint32_t dead,
                                                float (&scale)[8], int (&ex)[8])
{
    float mx[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) mx[r] = 0.f;
    for (int kb = 0; kb < kblocks; ++kb) {
        float q[8], u[8];
        fold_load_los<false>(S, list, kb, lane, src_of, q, u);
        fold_mask_los(S, kb, lane, dead, q, u);
#pragma unroll
        for (int r = 0; r < 8; ++r) mx[r] = fmaxf(mx[r], fmaxf(fabsf(q[r]), fabsf(u[r])));
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], o));
        ex[r] = fold_exponent(mx[r]);
        scale[r] = ldexpf(1.0f, ex[r]);
    }
}

// One K block of LOS r0 .. r0 + N - 1 of a group of 8, Q or U; rows: the group's first
// operand row in K block kb of the image.
template <int MODE, bool RING, int N>
__device__ __forceinline__ void fold_emit_rows(uint8_t *rows, int lane, int r0, const float (&v)[N], const float (&scale)[8])
{
    uint8_t *const mine = rows + ((lane & 1) ? kFoldPart : 0) + 4 * ((lane >> 1) & 3);
    const int chunk = lane >> 3;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int r = r0 + j;
        const uint32_t w = split_one<MODE>(MODE == MODE_FP16X3 ? v[j] * scale[j] : v[j]);
        const uint32_t p = __shfl_xor_sync(0xffffffffu, w, 1);
        const uint32_t o = (lane & 1) ? __byte_perm(p, w, 0x7632) : __byte_perm(w, p, 0x5410);
        uint8_t *at = mine + r * kFoldRowBytes + ((chunk ^ ((r >> 1) & 3)) << 4);
        const uint32_t store = MODE != MODE_BF16 || !(lane & 1);
        if (RING)
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t"
                         "@p st.global.L2::cache_hint.b32 [%0], %1, %2;\n\t}" ::"l"(at),
                         "r"(o), "l"(l2_evict_last()), "r"(store)
                         : "memory");
        else if (store)
            *reinterpret_cast<uint32_t *>(at) = o;
    }
}
