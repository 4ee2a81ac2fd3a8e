// Folded synthesis in one kernel (see fold.cu for the folded form and gemm.cu for
// the contraction): the layout stage runs inside the contraction's CTAs.
//
// As two kernels the operand image goes to HBM and back between them, 16 of the
// 24 bytes per (LOS, active channel) that a call moves besides F.  Here each CTA
// of a pair converts its own next 64 LOS while it contracts the current ones, into
// one of two slots of a small image ring that stays in L2 (2 tiles per CTA: 58 MB
// for 360 active channels; plain BF16, half as much a channel, see fused_prepare),
// and the TMA producer reads the slot once per phase tile.  The MMAs, their order
// and the scaling are gemm.cu's, so the results are the same bits.
//
// CTA pairs (cta_group::2), 640 threads per CTA:
//   warp 0      producer: TMA of the ring slot's operand and of the B hi/lo tiles -> full
//   warp 1      TMEM allocator, MMA issuer (one elected lane)    -> empty, tfull, afree
//   warp 2      loader (LOS-major): bulk copies of Q and U rows into staging slots -> sfull
//   warps 4-11  epilogue: warp w owns TMEM lane quarter w % 4 and column half
//               (w - 4) / 4; every phase tile is a single accumulation, so it goes
//               from TMEM straight to F and the running peak       -> tempty
//   warps 12-19 splitters: FP32 Q/U -> 16-bit hi/lo rows in the ring  -> sempty, ready
// Channel-major cubes load straight into the splitters' registers (a warp reads 128
// bytes of a channel row; bulk copies of 256-byte rows were slower, 0.83 against 0.43 ms
// without F on 262,144 LOS x 360 x 401).  LOS-major cubes come through staging slots of
// all channels of 8 LOS, one bulk copy per array, which leaves the channel gather to
// shared memory; where 8 rows do not fit, the base is not on 16 bytes, on a last, partial
// item, or with one item per pair, the splitters load through registers.  FP16X3 reads its
// exponents, a pass of their own before (fold.cu).
// 262,144 LOS x 360 x 401 with F: 0.505 ms a call on changing inputs under load, 0.454 ms on
// repeated ones at boost clocks.  Channel-major the splitters are busy 98% of the time (bound by
// the latency of loads whose channels lie a megabyte apart), the epilogue (F stores and the
// peak search) 78%, the MMAs 62%, most of that at the shared-memory bandwidth of their
// operands; LOS-major (0.455 ms) the MMAs 79%, slowed by the staging's traffic.  L2-evict-first
// loads and an evict-last ring keep the ring on chip: 6% of the call when they came.
// Every wait is bounded, as in gemm.cu.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <limits.h>

#include <algorithm>
#include <cstdlib>

#include "rms_internal.h"

namespace {

#include "tc_ptx.cuh"
#include "fold_split.cuh"

constexpr int kThreads = 640;
constexpr int kEpiWarp0 = 4, kNumEpiWarps = 8, kSplitWarp0 = 12, kNumSplitWarps = 8;
constexpr int kTmemCols = 512, kAccStride = 256;
constexpr int kMaxSlots = 3;                    // staging slots
constexpr int kSmemLimit = 227 * 1024;
// 640 x 96 registers: the epilogue takes them from the control and splitter warpgroups
constexpr int kRegsLaunch = 96, kRegsCtl = 48, kRegsEpi = 128, kRegsSplit = 88;
static_assert(128 * kRegsCtl + 256 * kRegsEpi + 256 * kRegsSplit == kThreads * kRegsLaunch,
              "register split must fill the launch");

constexpr int kMaxChunks = 4;

struct FusedParams {
    FoldSource src;
    int32_t kblocks, mode;
    int32_t nphi, ncol, kplus, kminus;
    int32_t ntiles_n, tile_n, tile_n_last, npad;
    uint8_t *ring;              // [CTAs][2][kblocks][parts x 8 KB]
    float *F;
    int32_t *pidx;
    float *pabs, *pphi, *pq, *pu, *pchi;
    const float *phi32;
    const double *phi64;
    double lambda0sq;
    float out_scale;
    const int8_t *rexp;         // FP16X3: [nlos] exponents
    int *err;
    int64_t timeout_ns;
    int32_t stages, kbs;        // pipeline stages of kbs K blocks each
    int32_t sslots;             // staging slots; 0: direct loads
    int32_t chunk_log;          // the splitters release an item's K blocks by parts of 2^chunk_log (>= kbs)
    uint32_t sbytes;            // bytes of a staging slot
    FusedRotation rot;          // ROT
};

__host__ __device__ __forceinline__ uint32_t sub_stage_bytes(int tile_n, int mode)
{
    const uint32_t parts = mode == MODE_BF16 ? 1u : 2u;
    return parts * (uint32_t)kFoldPart + parts * (uint32_t)(tile_n / 2) * kFoldRowBytes;
}

struct FSmem {
    uint8_t *ring, *stage;
    uint32_t stage_bytes, sub_bytes;
    float *pk_m, *pk_re, *pk_im;
    int *pk_i;
    int *list;                  // [kblocks x 32]: the padded channel list (an index load from L2 before
                                // every batch of data loads would double their latency)
    uint64_t *full, *empty, *tfull, *tempty, *ready, *afree, *sfull, *sempty, *pkfull, *pkempty, *mma_done;
    uint32_t *tmem_slot;
    volatile int *abort_flag;
};

__device__ __forceinline__ FSmem fcarve(uint8_t *base, const FusedParams &P)
{
    FSmem s;
    s.sub_bytes = sub_stage_bytes(P.tile_n, P.mode);
    s.stage_bytes = s.sub_bytes * (uint32_t)P.kbs;
    s.ring = base;
    s.stage = base + (size_t)P.stages * s.stage_bytes;
    s.pk_m = reinterpret_cast<float *>(s.stage + (size_t)P.sslots * P.sbytes);
    s.pk_i = reinterpret_cast<int *>(s.pk_m + 2 * 64);
    s.pk_re = reinterpret_cast<float *>(s.pk_i + 2 * 64);
    s.pk_im = s.pk_re + 2 * 64;
    s.list = reinterpret_cast<int *>(s.pk_im + 2 * 64);
    uint64_t *b = reinterpret_cast<uint64_t *>(s.list + P.kblocks * kKBlock);
    s.full = b;
    s.empty = s.full + P.stages;
    s.tfull = s.empty + P.stages;
    s.tempty = s.tfull + 2;
    s.ready = s.tempty + 2;
    s.afree = s.ready + 2 * kMaxChunks;
    s.sfull = s.afree + 2;
    s.sempty = s.sfull + kMaxSlots;
    s.pkfull = s.sempty + kMaxSlots;
    s.pkempty = s.pkfull + 8;
    s.mma_done = s.pkempty + 8;
    s.tmem_slot = reinterpret_cast<uint32_t *>(s.mma_done + 1);
    s.abort_flag = reinterpret_cast<volatile int *>(s.tmem_slot + 1);
    return s;
}
constexpr size_t kFixedSmem = 1024 + 8 * 64 * 4 + 8 * (2 * 3 + 2 * kMaxChunks + 2 * kMaxSlots + 16 + 1) + 16;

// 16 lanes x 32 consecutive 32-bit columns, no wait: four tmem_ld16x256 side by side.
__device__ __forceinline__ void tmem_ld16x256x4(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// Untiled bulk copy of data that is read once.
__device__ __forceinline__ void bulk_load_once(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(l2_evict_first())
                 : "memory");
}

// Channel-major tile, one splitter warp: 32 LOS (half of the tile), one array (Q or U), every
// other half K block of 16 channels, so that four warps share the work of a LOS.  f(h, v) gets
// the 16 values of half K block h; the next ones are loaded ahead.
template <bool LAST, typename F>
__device__ __forceinline__ void chan_walk(const FoldSource &S, const int *list, int64_t los, int array, int h0, int nh,
                                          F f)
{
    const float *const X = array ? S.U : S.Q;
    const bool valid = los < S.nlos;
    const int64_t at = min(los, S.nlos - 1);
    auto load = [&](int h, float (&v)[16]) {
        // unconditional loads (the channel list is padded with a valid channel), so that all
        // 16 are in flight at once
        int ch[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int4 c = *reinterpret_cast<const int4 *>(list + 16 * h + 4 * j);
            ch[4 * j] = c.x; ch[4 * j + 1] = c.y; ch[4 * j + 2] = c.z; ch[4 * j + 3] = c.w;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = load_here<LAST>(X + (int64_t)ch[j] * S.nlos + at);
    };
    auto masked = [&](int h, float (&v)[16]) {
        if (16 * h + 16 > S.nact || !valid) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (16 * h + j >= S.nact || !valid) v[j] = 0.f;
        }
        f(h, v);
    };
    float a[16], b[16];
    if (h0 < nh) load(h0, a);
    for (int h = h0; h < nh; h += 4) {
        if (h + 2 < nh) load(h + 2, b);
        masked(h, a);
        if (h + 4 < nh) load(h + 4, a);
        if (h + 2 < nh) masked(h + 2, b);
    }
}

// 64 bytes at a 32-byte aligned address
__device__ __forceinline__ void load64(const float *p, float (&v)[16])
{
#pragma unroll
    for (int h = 0; h < 2; ++h)
        asm volatile("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(v[8 * h]), "=f"(v[8 * h + 1]), "=f"(v[8 * h + 2]), "=f"(v[8 * h + 3]), "=f"(v[8 * h + 4]),
                       "=f"(v[8 * h + 5]), "=f"(v[8 * h + 6]), "=f"(v[8 * h + 7])
                     : "l"(p + 8 * h));
}

// (q + iu) t
__device__ __forceinline__ void rotate(float &q, float &u, float2 t)
{
    const float qr = fmaf(q, t.x, -u * t.y), ur = fmaf(q, t.y, u * t.x);
    q = qr;
    u = ur;
}

// ROT: window synthesis (learned.cu): every LOS is multiplied by its own row of T on its
// way into the ring, in FP32 like the data.
template <int MODE, bool CHAN, bool ROT>
__global__ void __launch_bounds__(kThreads, 1)
fused_kernel(const __grid_constant__ FusedParams P, const __grid_constant__ CUtensorMap tmB_hi,
             const __grid_constant__ CUtensorMap tmB_lo, const __grid_constant__ CUtensorMap tmA)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const FSmem S = fcarve(base, P);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr bool kSplitPrec = MODE != MODE_BF16;
    constexpr uint32_t kPartsBytes = (kSplitPrec ? 2 : 1) * kFoldPart;   // one K block of a ring slot
    const int64_t nlos = P.src.nlos;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const int64_t nit = (nlos + 2 * kFoldTileLos - 1) / (2 * kFoldTileLos);   // items: 64 LOS in each CTA
    const int64_t it0 = blockIdx.x >> 1, istride = gridDim.x >> 1;
    const uint32_t b_bytes = (uint32_t)(P.tile_n / 2) * kFoldRowBytes;
    const uint32_t peer_abort = mapa_shared(smem_u32((const void *)S.abort_flag), rank ^ 1u);
    auto stop_peer = [&]() { st_cluster_u32(peer_abort, 1u); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < P.stages; ++s) {
            mbar_init(smem_u32(&S.full[s]), 1);
            mbar_init(smem_u32(&S.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&S.tfull[b]), 1);
            mbar_init(smem_u32(&S.tempty[b]), 2 * kNumEpiWarps);
            for (int c = 0; c < kMaxChunks; ++c) mbar_init(smem_u32(&S.ready[b * kMaxChunks + c]), kNumSplitWarps);
            mbar_init(smem_u32(&S.afree[b]), 1);
        }
        for (int i = 0; i < 8; ++i) {
            mbar_init(smem_u32(&S.pkfull[i]), 1);
            mbar_init(smem_u32(&S.pkempty[i]), 1);
        }
        for (int i = 0; i < kMaxSlots; ++i) {
            mbar_init(smem_u32(&S.sfull[i]), 1);
            mbar_init(smem_u32(&S.sempty[i]), kNumSplitWarps);
        }
        mbar_init(smem_u32(S.mma_done), 1);
        *S.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < P.kblocks * kKBlock; i += kThreads) S.list[i] = P.src.padded[i];
    if (warp == 1) {
        __syncwarp();
        tmem_alloc_pair(smem_u32(S.tmem_slot), kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *S.tmem_slot;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCtl));
        if (warp == 0) {
            // ------------------------------------------------------------ producer
            if (lane == 0) {
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB_hi)) : "memory");
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB_lo)) : "memory");
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
                const uint32_t tx = kPartsBytes + (kSplitPrec ? 2 : 1) * b_bytes;
                int s = 0;
                uint32_t ph = 0, pending = 0, pend_par = 0;
                bool ok = true;
                int n_item = 0;
                for (int64_t it = it0; it < nit && ok; it += istride, ++n_item) {
                    const int slot = n_item & 1;
                    const int32_t z0 = ((int32_t)blockIdx.x * 2 + slot) * P.kblocks;
                    for (int nt = 0; nt < P.ntiles_n && ok; ++nt) {
                        int32_t y = nt * P.tile_n;
                        if (!leader) y += ((nt == P.ntiles_n - 1) ? P.tile_n_last : P.tile_n) / 2;
                        for (int kb = 0; kb < P.kblocks; kb += P.kbs) {
                            const int n = min(P.kbs, P.kblocks - kb);
                            if (nt == 0 && (kb & ((1 << P.chunk_log) - 1)) == 0) {
                                // the item's next K blocks are in the ring
                                if (!wait_bounded(smem_u32(&S.ready[slot * kMaxChunks + (kb >> P.chunk_log)]), (n_item >> 1) & 1,
                                                  S.abort_flag, P.err, P.timeout_ns)) {
                                    ok = false;
                                    break;
                                }
                                fence_proxy_async_global();
                            }
                            if (!wait_bounded(smem_u32(&S.empty[s]), ph ^ 1, S.abort_flag, P.err, P.timeout_ns)) {
                                ok = false;
                                break;
                            }
                            uint32_t st = smem_u32(S.ring + (size_t)s * S.stage_bytes);
                            const uint32_t bar = smem_u32(&S.full[s]);
                            const uint32_t bar0 = mapa_shared(bar, 0u);
                            if (leader) mbar_arrive_expect_tx(bar, 2 * tx * (uint32_t)n);
                            for (int i = 0; i < n; ++i, st += S.sub_bytes) {
                                tma_load_3d_pair(st, &tmA, 0, 0, z0 + kb + i, bar0);
                                const int32_t yb = ((kb + i) * P.npad + y) / kFoldMapRows;
                                tma_load_2d_pair(st + kPartsBytes, &tmB_hi, 0, yb, bar0);
                                if (kSplitPrec) tma_load_2d_pair(st + kPartsBytes + b_bytes, &tmB_lo, 0, yb, bar0);
                            }
                            pending |= 1u << s;
                            pend_par = (pend_par & ~(1u << s)) | (ph << s);
                            if (++s == P.stages) { s = 0; ph ^= 1; }
                        }
                    }
                }
                if (!ok) {
                    stop_peer();
                    if (leader) {
                        for (int i = 0; i < P.stages; ++i)
                            if (pending & (1u << i))
                                wait_bounded(smem_u32(&S.full[i]), (pend_par >> i) & 1, S.abort_flag, P.err,
                                             P.timeout_ns, false);
                    } else {
                        // the odd CTA's copies complete on the even CTA's barriers: give any still in
                        // flight far longer than a copy takes before this CTA may leave
                        const uint64_t t0 = global_ns();
                        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
                    }
                } else {
                    // the MMAs' commits arrive on this CTA's barriers from the tensor core: wait for
                    // the one that releases each slot's last fill before the CTA may exit
                    for (int i = 0; i < P.stages; ++i)
                        if ((pending & (1u << i)) &&
                            !wait_bounded(smem_u32(&S.empty[i]), (pend_par >> i) & 1, S.abort_flag, P.err,
                                          P.timeout_ns)) {
                            stop_peer();
                            break;
                        }
                }
            }
        } else if (warp == 1) {
            if (!leader) {
                // the even CTA's last commit: all MMAs that touch this CTA are complete
                if (lane == 0 && !wait_bounded(smem_u32(S.mma_done), 0, S.abort_flag, P.err, P.timeout_ns)) stop_peer();
            } else {
                // -------------------------------------------------------- MMA issuer
                const uint32_t one = elect_one();
                constexpr bool bf = MODE != MODE_FP16X3;
                const uint32_t id_full = idesc_f16_m(2 * kTileM, P.tile_n, bf);
                const uint32_t id_last = idesc_f16_m(2 * kTileM, P.tile_n_last, bf);
                int s = 0, g_all = 0, n_item = 0;
                uint32_t ph = 0, tph = 0;
                bool ok = true;
                auto arrived = [&](const uint64_t *bar, uint32_t parity) {
                    const bool in =
                        wait_bounded_cluster(smem_u32(bar), parity, S.abort_flag, P.err, P.timeout_ns);
                    return __all_sync(0xffffffffu, in) != 0;
                };
                for (int64_t it = it0; it < nit && ok; it += istride, ++n_item) {
                    for (int nt = 0; nt < P.ntiles_n && ok; ++nt, ++g_all) {
                        const uint32_t idesc = (nt == P.ntiles_n - 1) ? id_last : id_full;
                        const int b = g_all & 1;
                        if (!arrived(&S.tempty[b], ((tph >> b) & 1) ^ 1)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t d = tmem_base + (uint32_t)(b * kAccStride);
                        for (int kb = 0; kb < P.kblocks; kb += P.kbs) {
                            const int n = min(P.kbs, P.kblocks - kb);
                            if (!arrived(&S.full[s], ph)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            uint32_t st = smem_u32(S.ring + (size_t)s * S.stage_bytes);
                            for (int i = 0; i < n; ++i, st += S.sub_bytes) {
                                const uint32_t a_hi = st, a_lo = st + kFoldPart;
                                const uint32_t b_hi = st + kPartsBytes, b_lo = b_hi + b_bytes;
#pragma unroll
                                for (int kk = 0; kk < kKBlock / 16; ++kk) {
                                    const uint32_t ko = kk * 32;
                                    const uint32_t acc = (kb > 0 || i > 0 || kk > 0) ? 1u : 0u;
                                    mma_f16_pair(d, sdesc_k64(a_hi + ko), sdesc_k64(b_hi + ko), idesc, acc, one);
                                    if (kSplitPrec) {
                                        mma_f16_pair(d, sdesc_k64(a_hi + ko), sdesc_k64(b_lo + ko), idesc, 1u, one);
                                        mma_f16_pair(d, sdesc_k64(a_lo + ko), sdesc_k64(b_hi + ko), idesc, 1u, one);
                                    }
                                }
                            }
                            mma_commit_pair_mc(smem_u32(&S.empty[s]), (uint16_t)3, one);
                            if (++s == P.stages) { s = 0; ph ^= 1; }
                        }
                        if (!ok) break;
                        mma_commit_pair_mc(smem_u32(&S.tfull[b]), (uint16_t)3, one);
                        tph ^= 1u << b;
                    }
                    // every load of the item's ring slot has arrived (in both CTAs): the splitters may refill it
                    if (ok) mma_commit_pair_mc(smem_u32(&S.afree[n_item & 1]), (uint16_t)3, one);
                }
                if (!ok) stop_peer();
                // both CTAs wait for this commit before they leave (the odd CTA in its warp 1)
                mma_commit_pair_mc(smem_u32(S.mma_done), (uint16_t)3, one);
                wait_bounded(smem_u32(S.mma_done), 0, S.abort_flag, P.err, P.timeout_ns, false);
            }
        } else if (!CHAN && warp == 2 && P.sslots > 0) {
            // ------------------------------------------------------------ loader
            // 8 whole rows of each array per slot: [array][8][nchan]
            if (lane == 0) {
                const uint32_t bytes = 8u * (uint32_t)P.src.nchan * 4u;
                int s = 0;
                uint32_t ph = 0, pending = 0, pend_par = 0;
                bool ok = true;
                for (int64_t it = it0; it < nit && ok; it += istride) {
                    const int64_t los0 = (2 * it + rank) * kFoldTileLos;
                    if (los0 + kFoldTileLos > nlos) continue;      // the splitters load a partial item
                    for (int g = 0; g < kFoldTileLos / 8; ++g) {
                        if (!wait_bounded(smem_u32(&S.sempty[s]), ph ^ 1, S.abort_flag, P.err, P.timeout_ns)) {
                            ok = false;
                            break;
                        }
                        const uint32_t dst = smem_u32(S.stage + (size_t)s * P.sbytes), bar = smem_u32(&S.sfull[s]);
                        const int64_t at = (los0 + 8 * g) * P.src.nchan;
                        mbar_arrive_expect_tx(bar, 2 * bytes);
                        bulk_load_once(dst, P.src.Q + at, bytes, bar);
                        bulk_load_once(dst + bytes, P.src.U + at, bytes, bar);
                        pending |= 1u << s;
                        pend_par = (pend_par & ~(1u << s)) | (ph << s);
                        if (++s == P.sslots) { s = 0; ph ^= 1; }
                    }
                }
                if (!ok) stop_peer();
                // copies in flight land before the CTA may leave
                for (int i = 0; i < P.sslots; ++i)
                    if (pending & (1u << i))
                        wait_bounded(smem_u32(&S.sfull[i]), (pend_par >> i) & 1, S.abort_flag, P.err, P.timeout_ns, false);
            }
        }
    } else if (warp < kSplitWarp0) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        // ------------------------------------------------------------ epilogue
        // TMEM lanes and F's sectors as in gemm.cu: thread (rq, cq) holds the Q and U rows
        // of LOS 16 q + 8 l + rq, columns 4 g + cq; a lane whose sample lies in the next
        // 32-byte sector stores one group later.  32 columns of both LOS are loaded ahead.
        const int q = warp & 3, h = (warp - kEpiWarp0) >> 2;
        const int rq = lane >> 2, cq = lane & 3;
        uint32_t tph = 0;
        int g_all = 0, n_item = 0;
        bool ok = true;
        uint32_t tempty_addr[2];
        for (int b = 0; b < 2; ++b) tempty_addr[b] = mapa_shared(smem_u32(&S.tempty[b]), 0u);
        const int half = (P.tile_n / 16) * 8;          // columns of half 0 (a multiple of 8)
        for (int64_t it = it0; it < nit && ok; it += istride, ++n_item) {
            const int64_t row0 = (2 * it + rank) * kFoldTileLos + 16 * q + rq;
            float scale[2];
#pragma unroll
            for (int l = 0; l < 2; ++l)
                scale[l] = MODE == MODE_FP16X3 ? ldexpf(P.out_scale, -(int)__ldg(P.rexp + min(row0 + 8 * l, nlos - 1)))
                                               : P.out_scale;
            float bm[2] = {-1.f, -1.f}, br[2] = {0.f, 0.f}, bim[2] = {0.f, 0.f};
            int bi[2] = {INT_MAX, INT_MAX};
            for (int nt = 0; nt < P.ntiles_n; ++nt, ++g_all) {
                const int b = g_all & 1;
                if (!warp_wait(smem_u32(&S.tfull[b]), (tph >> b) & 1, S.abort_flag, P.err, P.timeout_ns)) {
                    ok = false;
                    break;
                }
                tph ^= 1u << b;
                tc_fence_after();
                const int ncols = ((nt == P.ntiles_n - 1) ? P.tile_n_last : P.tile_n) - h * half;
                const int kbase = (nt * P.tile_n + h * half) >> 1;
                const int mine = min(ncols, h ? P.tile_n - half : half);   // columns of this half with results
                const uint32_t taddr = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * kAccStride + h * half);
                float2 *dp[2], *dm[2];
                bool latep[2], latem[2], st[2];
                float2 prevp[2], prevm[2];
                bool okp1 = false, okm1 = false;
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const int64_t r = row0 + 8 * l;
                    st[l] = P.F != nullptr && r < nlos;
                    dp[l] = reinterpret_cast<float2 *>(P.F) + (r * P.nphi + P.kplus + kbase);
                    dm[l] = reinterpret_cast<float2 *>(P.F) + (r * P.nphi + P.kminus - kbase);
                    latep[l] = (int)((reinterpret_cast<uintptr_t>(dp[l]) >> 3) & 3) + cq >= 4;
                    latem[l] = (int)((reinterpret_cast<uintptr_t>(dm[l]) >> 3) & 3) < cq;
                    dp[l] += cq - (latep[l] ? 4 : 0);
                    dm[l] -= cq - (latem[l] ? 4 : 0);
                    prevp[l] = prevm[l] = make_float2(0.f, 0.f);
                }
                auto group = [&](int gg, const uint32_t (&v0)[4], const uint32_t (&v1)[4], bool last) {
                    // last: no columns of its own, only the late lanes' stores of the group before
                    const int c = kbase + 4 * gg + cq;
                    const bool ok2 = !last && 2 * (4 * gg + cq) < mine && c < P.ncol;
                    const bool okp = ok2 && (!ROT || P.kplus + c < P.nphi);    // a window has one -phi sample more
                    const bool okm = ok2 && P.kminus - c != P.kplus + c;       // phi = 0 is its own partner
#pragma unroll
                    for (int l = 0; l < 2; ++l) {
                        const uint32_t(&v)[4] = l ? v1 : v0;
                        const float qc = __uint_as_float(v[0]), qs = __uint_as_float(v[1]);
                        const float uc = __uint_as_float(v[2]), us = __uint_as_float(v[3]);
                        const float2 vp = make_float2((qc + us) * scale[l], (uc - qs) * scale[l]);
                        const float2 vm = make_float2((qc - us) * scale[l], (uc + qs) * scale[l]);
                        const float mp = __fadd_rn(__fmul_rn(vp.x, vp.x), __fmul_rn(vp.y, vp.y));
                        const float mm = __fadd_rn(__fmul_rn(vm.x, vm.x), __fmul_rn(vm.y, vm.y));
                        // lowest index among equals: a +phi index is above, a -phi one below all before it
                        if (okp && mp > bm[l]) { bm[l] = mp; bi[l] = P.kplus + c; br[l] = vp.x; bim[l] = vp.y; }
                        if (okm && mm >= bm[l]) { bm[l] = mm; bi[l] = P.kminus - c; br[l] = vm.x; bim[l] = vm.y; }
                        if (st[l]) {
                            // streaming stores: F is written once and must not push the operands out of L2
                            if (latep[l] ? okp1 : okp) __stcs(dp[l] + 4 * gg, latep[l] ? prevp[l] : vp);
                            if (latem[l] ? okm1 : okm) __stcs(dm[l] - 4 * gg, latem[l] ? prevm[l] : vm);
                        }
                        prevp[l] = vp;
                        prevm[l] = vm;
                    }
                    okp1 = okp;
                    okm1 = okm;
                };
                for (int c0 = 0; c0 < mine; c0 += 32) {
                    uint32_t v[2][16];
                    __syncwarp();       // (lanes may have parted over the stores and peaks of the columns before)
                    tmem_ld16x256x4(taddr + c0, v[0]);
                    tmem_ld16x256x4(taddr + (16u << 16) + c0, v[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (c0 + 8 * j >= mine) break;
                        const uint32_t a0[4] = {v[0][4 * j], v[0][4 * j + 1], v[0][4 * j + 2], v[0][4 * j + 3]};
                        const uint32_t a1[4] = {v[1][4 * j], v[1][4 * j + 1], v[1][4 * j + 2], v[1][4 * j + 3]};
                        group((c0 >> 3) + j, a0, a1, false);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(tempty_addr[b]);
                const uint32_t none[4] = {0u, 0u, 0u, 0u};
                if (mine > 0) group((mine + 7) >> 3, none, none, true);
            }
            if (!ok) break;
            // the four lanes of a row group hold disjoint columns of the same two LOS: a butterfly
            // leaves every lane with both peaks (lowest index on ties); lane cq owns LOS l = cq
#pragma unroll
            for (int l = 0; l < 2; ++l)
#pragma unroll
                for (int off = 1; off <= 2; off <<= 1) {
                    const float om = __shfl_xor_sync(0xffffffffu, bm[l], off);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi[l], off);
                    const float ore = __shfl_xor_sync(0xffffffffu, br[l], off);
                    const float oim = __shfl_xor_sync(0xffffffffu, bim[l], off);
                    if (om > bm[l] || (om == bm[l] && oi < bi[l])) { bm[l] = om; bi[l] = oi; br[l] = ore; bim[l] = oim; }
                }
            const bool owner = cq < 2;
            float pm = cq ? bm[1] : bm[0], pre = cq ? br[1] : br[0], pim = cq ? bim[1] : bim[0];
            int pi = cq ? bi[1] : bi[0];
            // combine the two column halves: half 1 publishes, half 0 writes
            const int par = n_item & 1, at = par * 64 + 16 * q + 8 * (cq & 1) + rq;
            const uint32_t pbar = smem_u32(&S.pkfull[par * 4 + q]), ebar = smem_u32(&S.pkempty[par * 4 + q]);
            const uint32_t use_par = (n_item >> 1) & 1;
            if (h == 1) {
                if (!warp_wait(ebar, use_par ^ 1, S.abort_flag, P.err, P.timeout_ns)) { ok = false; break; }
                if (owner) {
                    S.pk_m[at] = pm;
                    S.pk_i[at] = pi;
                    S.pk_re[at] = pre;
                    S.pk_im[at] = pim;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(pbar);
            } else {
                if (!warp_wait(pbar, use_par, S.abort_flag, P.err, P.timeout_ns)) { ok = false; break; }
                const float om = S.pk_m[at], ore = S.pk_re[at], oim = S.pk_im[at];
                const int oi = S.pk_i[at];
                __syncwarp();
                if (lane == 0) mbar_arrive(ebar);
                if (om > pm || (om == pm && oi < pi)) { pm = om; pi = oi; pre = ore; pim = oim; }
                const int64_t r = (2 * it + rank) * kFoldTileLos + 16 * q + 8 * (cq & 1) + rq;
                if (owner && r < nlos) {
                    const bool found = pi != INT_MAX;
                    const float nan = __int_as_float(0x7fc00000);
                    if (P.pidx) P.pidx[r] = found ? pi : -1;
                    if (P.pabs) P.pabs[r] = found ? sqrtf(pm) : nan;
                    if (P.pphi) P.pphi[r] = found ? P.phi32[pi] : nan;
                    if (P.pq) P.pq[r] = found ? pre : nan;
                    if (P.pu) P.pu[r] = found ? pim : nan;
                    if (P.pchi) {
                        // chi0 = arg F(phi_peak) / 2 - phi_peak lambda_0^2, reduced to [0, pi)
                        float c = nan;
                        if (found) {
                            double x = 0.5 * atan2((double)pim, (double)pre) - P.phi64[pi] * P.lambda0sq;
                            x -= M_PI * floor(x / M_PI);
                            c = (float)x;
                        }
                        P.pchi[r] = c;
                    }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsSplit));
        // ------------------------------------------------------------ splitters
        const int sw = warp - kSplitWarp0;
        // channel-major: this warp's 32 LOS of the tile, its array and first half K block
        const int i = 32 * (sw & 1) + lane, array = (sw >> 1) & 1, h0 = sw >> 2;
        const int row = 16 * (i >> 3) + (i & 7) + 8 * array, swz = (row >> 1) & 3;
        int n_item = 0, ss = 0;
        uint32_t sph = 0;
        bool ok = true;
        for (int64_t it = it0; it < nit && ok; it += istride, ++n_item) {
            const int slot = n_item & 1;
            const int64_t los0 = (2 * it + rank) * kFoldTileLos;
            const bool stg = !CHAN && P.sslots > 0 && los0 + kFoldTileLos <= nlos;
            uint8_t *const tile = P.ring + ((size_t)blockIdx.x * 2 + slot) * P.kblocks * kPartsBytes;
            const int64_t los8 = los0 + 8 * sw;            // LOS-major, direct: this warp's 8 LOS
            auto src_of = [&](int r) { return min(los8 + r, nlos - 1); };
            const uint32_t dead = los8 + 8 <= nlos ? 0u : (0xffu << (int)max((int64_t)0, nlos - los8)) & 0xffu;
            // FP16X3: the exponents of the item's LOS, two per lane
            int e64[2] = {0, 0};
            if constexpr (MODE == MODE_FP16X3) {
#pragma unroll
                for (int h = 0; h < 2; ++h) e64[h] = __ldg(P.rexp + min(los0 + 32 * h + lane, nlos - 1));
            }
            // the scales of LOS j + 2 k + (lane / 16) of the item (j a multiple of 8)
            auto scales_of = [&](int j, float (&scale)[4]) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    scale[k] = MODE != MODE_FP16X3 ? 1.f
                               : ldexpf(1.0f, __shfl_sync(0xffffffffu, j & 32 ? e64[1] : e64[0], (j & 31) + 2 * k + (lane >> 4)));
            };
            float scale[4];
            // ROT: the T rows of the item's LOS, two LOS per lane, or the lane's own LOS (channel-major)
            int32_t cen[2] = {0, 0};
            if constexpr (ROT) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    cen[h] = max(P.rot.cmin, min(P.rot.cmax, __ldg(P.rot.centre + min(los0 + 32 * h + lane, nlos - 1))));
                if constexpr (CHAN) cen[0] = (sw & 1) ? cen[1] : cen[0];
            }
            // T of LOS j + (lane / 16) of the item (j even) at this lane's two channels of K block kb
            auto t_of = [&](int j, int kb) {
                const int c = __shfl_sync(0xffffffffu, j & 32 ? cen[1] : cen[0], (j & 31) + (lane >> 4));
                return __ldg(reinterpret_cast<const float4 *>(P.rot.T + (size_t)c * P.rot.ldT + kb * kKBlock) + (lane & 15));
            };
            // the slot's previous item has been read
            if (!warp_wait(smem_u32(&S.afree[slot]), ((n_item >> 1) & 1) ^ 1, S.abort_flag, P.err, P.timeout_ns)) {
                ok = false;
                break;
            }
            // release part c of the item's K blocks, as far as this warp goes
            auto release = [&](int c) {
                // the TMA (async proxy) reads what these generic stores wrote
                fence_proxy_async_global();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&S.ready[slot * kMaxChunks + c]));
            };
            if constexpr (CHAN) {
                if constexpr (ROT) {
                    // both arrays of 8 channels at a time; four warps share a LOS
                    const float2 *T = P.rot.T + (size_t)cen[0] * P.rot.ldT;
                    const int64_t at = min(los0 + i, nlos - 1);
                    const bool valid = los0 + i < nlos;
                    const int r0 = 16 * (i >> 3) + (i & 7), sz = (r0 >> 1) & 3;
                    auto load = [&](int o, float (&q)[8], float (&u)[8]) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int64_t off = (int64_t)S.list[8 * o + j] * nlos + at;
                            q[j] = load_here<true>(P.src.Q + off);
                            u[j] = load_here<true>(P.src.U + off);
                        }
                    };
                    // T of octet o at this LOS, in two loads of 32 bytes: every lane has a row (and a
                    // cache line per load) of its own
                    float t[16];
                    auto load_t = [&](int o) { load64(reinterpret_cast<const float *>(T + 8 * o), t); };
                    auto work = [&](int o, int next, float (&q)[8], float (&u)[8]) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (8 * o + j >= P.src.nact || !valid) q[j] = u[j] = 0.f;
                            rotate(q[j], u[j], make_float2(t[2 * j], t[2 * j + 1]));
                        }
                        load_t(next);
                        uint32_t qh[4], ql[4], uh[4], ul[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            split_pair_bf16(q[2 * j], q[2 * j + 1], qh[j], ql[j]);
                            split_pair_bf16(u[2 * j], u[2 * j + 1], uh[j], ul[j]);
                        }
                        uint8_t *d = tile + (size_t)(o >> 2) * kPartsBytes + r0 * kFoldRowBytes + (((o & 3) ^ sz) << 4);
                        *reinterpret_cast<uint4 *>(d) = make_uint4(qh[0], qh[1], qh[2], qh[3]);
                        *reinterpret_cast<uint4 *>(d + 8 * kFoldRowBytes) = make_uint4(uh[0], uh[1], uh[2], uh[3]);
                        if (kSplitPrec) {
                            *reinterpret_cast<uint4 *>(d + kFoldPart) = make_uint4(ql[0], ql[1], ql[2], ql[3]);
                            *reinterpret_cast<uint4 *>(d + kFoldPart + 8 * kFoldRowBytes) = make_uint4(ul[0], ul[1], ul[2], ul[3]);
                        }
                    };
                    // a warp's octets are one to a K block; the next one's values and T are in flight (whole
                    // 32-byte sectors, two octets at a time, leave no registers for that: 1,048,576 LOS
                    // learned peak map 5.24 ms, against 5.01 this way and 5.38 with nothing ahead)
                    constexpr int kStep = kNumSplitWarps / 2;
                    static_assert(kStep == 4, "one octet of every K block per warp");
                    for (int c = 0; c << P.chunk_log < P.kblocks; ++c) {
                        const int o1 = 4 * min(P.kblocks, (c + 1) << P.chunk_log), last = o1 - kStep + (sw >> 1);
                        float qa[8], ua[8], qb[8], ub[8];
                        int o = (4 * c << P.chunk_log) + (sw >> 1);
                        load_t(o);
                        load(o, qa, ua);
                        for (; o < o1; o += 2 * kStep) {
                            if (o + kStep < o1) load(o + kStep, qb, ub);
                            work(o, min(o + kStep, last), qa, ua);
                            if (o + 2 * kStep < o1) load(o + 2 * kStep, qa, ua);
                            if (o + kStep < o1) work(o + kStep, min(o + 2 * kStep, last), qb, ub);
                        }
                        release(c);
                    }
                } else {
                uint8_t *const dst = tile + row * kFoldRowBytes;
                const float sc = MODE == MODE_FP16X3 ? ldexpf(1.0f, sw & 1 ? e64[1] : e64[0]) : 1.f;
                for (int c = 0; c << P.chunk_log < P.kblocks; ++c) {
                    const int h1 = 2 * min(P.kblocks, (c + 1) << P.chunk_log);
                    chan_walk<true>(P.src, S.list, los0 + i, array, (2 * c << P.chunk_log) + h0, h1, [&](int h, const float (&v)[16]) {
                        emit16<MODE, true>(dst + (size_t)(h >> 1) * kPartsBytes, h & 1, swz, v, sc);
                    });
                    release(c);
                }
                }
            } else if (stg) {
                // 8 LOS per slot; units of (K block, array), or ROT (K block, 4 LOS), go round the warps
                float4 t[2];
                if constexpr (ROT) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) t[j] = t_of(4 * (sw & 1) + 2 * j, min(sw >> 1, P.kblocks - 1));
                }
                for (int g = 0; g < kFoldTileLos / 8; ++g) {
                    if (!warp_wait(smem_u32(&S.sfull[ss]), sph, S.abort_flag, P.err, P.timeout_ns)) {
                        ok = false;
                        break;
                    }
                    const float *rows = reinterpret_cast<const float *>(S.stage + (size_t)ss * P.sbytes);
                    const int nchan = P.src.nchan;
                    if constexpr (MODE == MODE_FP16X3) scales_of(8 * g, scale);
                    const int arr = sw & 1;
                    for (int kb = sw >> 1; kb < P.kblocks; kb += kNumSplitWarps / 2) {
                        const int2 ch = *reinterpret_cast<const int2 *>(S.list + kb * kKBlock + 2 * (lane & 15));
                        const int left = P.src.nact - kb * kKBlock - 2 * (lane & 15);   // padding channels give 0
                        const int half = lane >> 4;
                        // the two halves read rows nchan words apart: with an even nchan the upper half
                        // takes its odd channels first, which keeps the 32 lanes on 32 banks
                        const bool flip = half && !(nchan & 1);
                        const int c0 = flip ? ch.y : ch.x, c1 = flip ? ch.x : ch.y;
                        auto pair_of = [&](const float *x, float &v0, float &v1) {
                            const float a = x[c0], b = x[c1];
                            v0 = left > 0 ? (flip ? b : a) : 0.f;
                            v1 = left > 1 ? (flip ? a : b) : 0.f;
                        };
                        uint8_t *const blk = tile + (size_t)kb * kPartsBytes + 16 * g * kFoldRowBytes;
                        if constexpr (ROT) {
                            const int r0 = 4 * arr;
                            const float one2[2] = {1.f, 1.f};       // (never FP16X3)
                            float q[4], u[4];
                            float4 tn[2];
                            // T of the warp's next unit, here or in the next slot
                            const bool more = kb + kNumSplitWarps / 2 < P.kblocks;
                            const int gn = more ? g : min(g + 1, kFoldTileLos / 8 - 1);
                            const int kn = more ? kb + kNumSplitWarps / 2 : sw >> 1;     // (kb itself is one: in range)
#pragma unroll
                            for (int j = 0; j < 2; ++j) tn[j] = t_of(8 * gn + r0 + 2 * j, kn);
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                const float *x = rows + (r0 + 2 * j + half) * nchan, *y = x + 8 * nchan;
                                pair_of(x, q[2 * j], q[2 * j + 1]);
                                pair_of(y, u[2 * j], u[2 * j + 1]);
                                rotate(q[2 * j], u[2 * j], make_float2(t[j].x, t[j].y));
                                rotate(q[2 * j + 1], u[2 * j + 1], make_float2(t[j].z, t[j].w));
                                t[j] = tn[j];
                            }
                            fold_emit_rows<MODE, true, 4>(blk, lane, r0, q, one2);
                            fold_emit_rows<MODE, true, 4>(blk + 8 * kFoldRowBytes, lane, r0, u, one2);
                        } else {
                            float v[8];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                pair_of(rows + (8 * arr + 2 * j + half) * nchan, v[2 * j], v[2 * j + 1]);
                            }
                            fold_emit_rows<MODE, true, 8>(blk + 8 * arr * kFoldRowBytes, lane, 0, v, scale);
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&S.sempty[ss]));
                    if (++ss == P.sslots) { ss = 0; sph ^= 1; }
                }
            } else {
                if constexpr (MODE == MODE_FP16X3) scales_of(8 * sw, scale);
                uint8_t *const dst = tile + 16 * sw * kFoldRowBytes;
                if constexpr (ROT || MODE == MODE_FP16X3) {
                    // one K block at a time: with the next one's values the registers run out here
                    for (int c = 0; ROT ? c < 1 : c << P.chunk_log < P.kblocks; ++c) {      // (ROT: one part)
                        const int kb1 = ROT ? P.kblocks : min(P.kblocks, (c + 1) << P.chunk_log);
#pragma unroll (ROT ? 1 : 2)
                        for (int kb = ROT ? 0 : c << P.chunk_log; kb < kb1; ++kb) {
                            float q[8], u[8];
                            fold_load_los<true>(P.src, S.list, kb, lane, src_of, q, u);
                            fold_mask_los(P.src, kb, lane, dead, q, u);
                            if constexpr (ROT) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    const float4 t = t_of(8 * sw + 2 * j, kb);
                                    rotate(q[2 * j], u[2 * j], make_float2(t.x, t.y));
                                    rotate(q[2 * j + 1], u[2 * j + 1], make_float2(t.z, t.w));
                                }
                            }
                            fold_emit_rows<MODE, true, 8>(dst + (size_t)kb * kPartsBytes, lane, 0, q, scale);
                            fold_emit_rows<MODE, true, 8>(dst + (size_t)kb * kPartsBytes + 8 * kFoldRowBytes, lane, 0, u, scale);
                        }
                        release(c);
                    }
                } else {
                    auto load = [&](int kb, float (&q)[8], float (&u)[8]) {
                        fold_load_los<true>(P.src, S.list, kb, lane, src_of, q, u);
                    };
                    auto emit = [&](int kb, float (&q)[8], float (&u)[8]) {
                        fold_mask_los(P.src, kb, lane, dead, q, u);
                        fold_emit_rows<MODE, true, 8>(dst + (size_t)kb * kPartsBytes, lane, 0, q, scale);
                        fold_emit_rows<MODE, true, 8>(dst + (size_t)kb * kPartsBytes + 8 * kFoldRowBytes, lane, 0, u, scale);
                    };
                    for (int c = 0; c << P.chunk_log < P.kblocks; ++c) {
                        const int kb1 = min(P.kblocks, (c + 1) << P.chunk_log);
                        float qa[8], ua[8], qb[8], ub[8];
                        int kb = c << P.chunk_log;
                        load(kb, qa, ua);
                        // the next K block's loads are in flight while one is split
                        for (; kb < kb1; kb += 2) {
                            if (kb + 1 < kb1) load(kb + 1, qb, ub);
                            emit(kb, qa, ua);
                            if (kb + 2 < kb1) load(kb + 2, qa, ua);
                            if (kb + 1 < kb1) emit(kb + 1, qb, ub);
                        }
                        release(c);
                    }
                }
            }
            if (!ok) break;
            if (stg) release(0);            // (one part)
        }
        // the commits that free the last slots arrive before the CTA leaves
        for (int k = max(0, n_item - 2); k < n_item && ok; ++k)
            ok = warp_wait(smem_u32(&S.afree[k & 1]), (k >> 1) & 1, S.abort_flag, P.err, P.timeout_ns);
        if (!ok) stop_peer();
        // the ring's lines go back to normal priority: nobody else's working set should yield to them.
        // (Here, beside the last epilogue: after it, it took 1.4 us of a 27 us call.)
        uint8_t *const own = P.ring + (size_t)blockIdx.x * 2 * P.kblocks * kPartsBytes;
        const uint32_t used = (uint32_t)min(n_item, 2) * P.kblocks * kPartsBytes;
        for (uint32_t at = (uint32_t)(32 * sw + lane) * 128; at < used; at += kNumSplitWarps * 32 * 128)
            asm volatile("applypriority.global.L2::evict_normal [%0], 128;" ::"l"(own + at) : "memory");
    }

    if (*S.abort_flag) stop_peer();
    tc_fence_before();
    __syncthreads();
    // neither CTA leaves (or frees TMEM) while the other may still use its shared memory,
    // barriers or TMEM
    cluster_sync_all();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace

namespace {

using FusedKernel = void (*)(FusedParams, CUtensorMap, CUtensorMap, CUtensorMap);

FusedKernel fused_for(int mode, bool chan, bool rot)
{
    if (rot) {      // window plans are BF16 or BF16X3
        if (mode == MODE_BF16) return chan ? fused_kernel<MODE_BF16, true, true> : fused_kernel<MODE_BF16, false, true>;
        return chan ? fused_kernel<MODE_BF16X3, true, true> : fused_kernel<MODE_BF16X3, false, true>;
    }
    if (mode == MODE_BF16) return chan ? fused_kernel<MODE_BF16, true, false> : fused_kernel<MODE_BF16, false, false>;
    if (mode == MODE_BF16X3) return chan ? fused_kernel<MODE_BF16X3, true, false> : fused_kernel<MODE_BF16X3, false, false>;
    return chan ? fused_kernel<MODE_FP16X3, true, false> : fused_kernel<MODE_FP16X3, false, false>;
}

// Pipeline shape beside `staging` bytes of staging slots and the channel list: K blocks per stage and stages, at
// least three of them; stages = 0 if they do not fit.
struct Shape {
    int kbs = 0, stages = 0;
    size_t smem = 0;
};
Shape shape_for(const rms_plan_s &p, size_t staging)
{
    Shape s;
    const int tile_n = p.fold.tiles.tile_n2, mode = mode_of(p.precision);
    staging += (size_t)p.fold.kpad * sizeof(int);
    for (s.kbs = 4; s.kbs >= 1; s.kbs /= 2) {
        const size_t per = s.kbs * (size_t)sub_stage_bytes(tile_n, mode) + 16;
        if (kFixedSmem + staging + 3 * per > (size_t)kSmemLimit) continue;
        s.stages = (int)std::min<size_t>(8, (kSmemLimit - kFixedSmem - staging) / per);
        s.smem = kFixedSmem + staging + s.stages * per;
        break;
    }
    return s;
}

// Staging slots of a LOS-major call: as many rows of 8 LOS as fit in 72 KB, two at least;
// none where the bulk copies' 16-byte rule does not hold.
constexpr size_t kStaging = 72 * 1024;
int staging_slots(const rms_plan_s &p, const float *Q, const float *U, bool chan)
{
    if (chan || ((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(U)) & 15)) return 0;
    const size_t slot = (size_t)2 * 8 * p.nchan * sizeof(float);
    return 2 * slot > kStaging ? 0 : (int)std::min<size_t>(kMaxSlots, kStaging / slot);
}

cudaLaunchConfig_t launch_config(cudaLaunchAttribute *attr, unsigned grid, size_t smem, cudaStream_t s)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(kThreads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = 2;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

}  // namespace

// Plans whose K blocks form one accumulation: 16 of 32 channels for the split precisions, any
// number for plain BF16.  Its ring is 8 KB per K block and slot, 2.4 MB per K block over 76
// pairs: 61 MB at 800 channels, 117 at 1,536, beyond the 129 MB L2 from 1,700 on.  The form pays to
// there and, without F, beyond; with F two kernels are up to 12 % faster on longer
// channel lists (not taken: the one-kernel form is still the faster one on single rounds there,
// 9,000 LOS x 2500 81 against 94 us).  One kernel against two, ms, channel-major with F / without:
// 262,144 LOS x 1000 x 401 0.83 / 0.93 and 0.66 / 0.85, x 1536 1.24 / 1.34 and 1.10 / 1.27, x 2000 1.69 /
// 1.72 and 1.56 / 1.64, x 2600 2.24 / 2.19 and 2.13 / 2.15, 93,568 x 2000 x 1601 1.25 / 1.21 and 1.03 /
// 1.14, 46,720 x 4000 x 1601 1.26 / 1.12 and 1.15 / 1.24, 262,144 x 1536 x 4001 5.29 / 4.96; LOS-major with F
// x 1536 1.23 / 1.27, x 2000 1.72 / 1.64, x 2600 2.33 / 2.12.
cudaError_t fused_prepare(rms_plan_s *p, bool window)
{
    FoldPlan &f = p->fold;
    f.fused_pairs = 0;
    const int mode = mode_of(p->precision);
    if (!f.pair_maps || (window && mode == MODE_FP16X3) || (mode != MODE_BF16 && f.kblocks > kGroupKBlocks)) return cudaSuccess;
    if (shape_for(*p, kStaging).stages < 3) return cudaSuccess;
    for (bool chan : {true, false}) {
        const FusedKernel k = fused_for(mode, chan, window);
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess && fa.numRegs != kRegsLaunch) e = cudaErrorInvalidConfiguration;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = launch_config(&attr, 2 * (p->num_sms / 2), kSmemLimit, 0);
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        if (e != cudaSuccess) return e;
        n = std::min(n, p->num_sms / 2);
        f.fused_pairs = chan ? n : std::min(f.fused_pairs, n);
    }
    return cudaSuccess;
}

// One kernel unless the last round of items over the pairs is too empty (12,000 LOS are 94
// items on 76 pairs: 69.9 against 64.2 us at 360 channels x 801 phi, but 161 items on two
// thirds of three rounds 89 against 97, LOS-major 100 against 95) or there are few items with
// many phase tiles, which the job schedule spreads over more SMs.  One kernel against two
// with F and the peak map, repeated inputs at boost clocks: 262,144 LOS x 360 x 401 BF16x3
// 0.454 / 0.604 ms (LOS-major 0.455 / 0.610), FP16x3 0.583 / 0.730, 200,003 x 357 LOS-major FP16x3
// 0.466 / 0.581, 400,000 x 800 x 1001 BF16 1.47 / 2.03 ms, 5,001 x 357 x 401 26.7 / 37.1 us; and at
// the line: 13,900 to 16,000 LOS x 401 0.73 to 0.89 of two kernels' time over 100 to 400 channels and
// all three precisions, 20,000 (69% of three rounds) 0.78 to 0.98 (1,200 channels BF16 1.00 to 1.04),
// 100 LOS x 1200 x 401 BF16 1.08 to 1.12 (fewer, longer items: a serial K).
bool fused_wanted(const rms_plan_s &p, int64_t nlos)
{
    const FoldPlan &f = p.fold;
    // options and knobs of the contraction kernel take a call there
    static const bool knobs = [] {
        for (const char *v : {"RMS_GEMM_PAIR", "RMS_GEMM_CTAS", "RMS_L2_BUDGET_MB", "RMS_GROUP_KBLOCKS", "RMS_MAX_TILE_N"})
            if (std::getenv(v)) return true;
        return false;
    }();
    if (f.fused_pairs < 1 || p.contraction != RMS_CONTRACT_AUTO || p.schedule != RMS_SCHEDULE_AUTO || p.l2_budget != 0 || knobs)
        return false;
    const int64_t nit = (nlos + 2 * kFoldTileLos - 1) / (2 * kFoldTileLos);
    const int64_t rounds = (nit + f.fused_pairs - 1) / f.fused_pairs;
    if (rounds == 1) return 2 * nit >= f.fused_pairs || f.tiles.ntiles_n2 <= 2;
    return 3 * nit >= 2 * rounds * f.fused_pairs;
}

size_t fused_ring_bytes(const rms_plan_s &p, int64_t nlos)
{
    const int64_t nit = (nlos + 2 * kFoldTileLos - 1) / (2 * kFoldTileLos);
    const size_t parts = p.precision == RMS_BF16 ? 1 : 2;
    return (size_t)(4 * std::min<int64_t>(nit, p.fold.fused_pairs)) * p.fold.kblocks * parts * kFoldPart;
}

cudaError_t launch_fused(const rms_plan_s &p, const float *Q, const float *U, int64_t nlos, int layout, float *F,
                         int32_t *pidx, float *pabs, float *pphi, float *pq, float *pu, float *pchi, uint8_t *ring,
                         const int8_t *rexp, cudaStream_t s, const FusedRotation *rot, CallFacts *facts)
{
    const FoldPlan &f = p.fold;
    const bool chan = layout == RMS_CHAN_MAJOR;
    const int mode = mode_of(p.precision);
    const int64_t nit = (nlos + 2 * kFoldTileLos - 1) / (2 * kFoldTileLos);
    const int pairs = (int)std::min<int64_t>(nit, f.fused_pairs);
    FusedParams P;
    P.src = {Q, U, nlos, p.nchan, p.nact, chan, p.d_active, f.d_list};
    P.kblocks = f.kblocks;
    P.mode = mode;
    if (rot) P.rot = *rot;
    P.nphi = p.nphi;
    P.ncol = f.ncol;
    P.kplus = f.kplus;
    P.kminus = f.kminus;
    P.ntiles_n = f.tiles.ntiles_n2;
    P.tile_n = f.tiles.tile_n2;
    P.tile_n_last = f.tiles.tile_n_last2;
    P.npad = f.tiles.npad;
    P.ring = ring;
    P.F = F;
    P.pidx = pidx;
    P.pabs = pabs;
    P.pphi = pphi;
    P.pq = pq;
    P.pu = pu;
    P.pchi = pchi;
    P.phi32 = p.d_phi32;
    P.phi64 = p.d_phi;
    P.lambda0sq = p.lambda0sq;
    P.out_scale = (float)(p.K * p.wmax);
    P.rexp = rexp;
    P.err = p.d_err;
    P.timeout_ns = p.timeout_ns;
    // One item per pair: its K blocks are released in up to four parts, so that the MMAs start while it
    // is being split; LOS-major it is then loaded K block by K block, not by whole staged rows (the
    // window's rows stay staged: its rotation leaves no registers for the loads ahead).  5,001 LOS x 357 x
    // 401 BF16x3 32.5 -> 27.1 us (channel-major 30.8 -> 26.7), 2,000 LOS 28.8 -> 24.7, 9,728 33.0 -> 28.8.
    // Fewer than five K blocks are one part: a part costs a fence and its loads' latency.
    const bool once = nit <= f.fused_pairs && (chan || !rot);
    P.sslots = once ? 0 : staging_slots(p, Q, U, chan);
    P.sbytes = (uint32_t)(2 * 8 * p.nchan * sizeof(float));
    const Shape sh = shape_for(p, (size_t)P.sslots * P.sbytes);
    if (sh.stages < 3) return cudaErrorInvalidConfiguration;
    P.stages = sh.stages;
    P.kbs = sh.kbs;
    for (P.chunk_log = 2; f.kblocks > (once ? kMaxChunks : 1) << P.chunk_log;) ++P.chunk_log;   // (4 >= kbs)
    // the ring as a 3-D tensor: 8 of the image's 64-byte rows to a row (whole lines per request), the
    // hi (and lo) rows of a K block, K blocks
    const int parts = mode == MODE_BF16 ? 1 : 2;
    constexpr int kRow = kFoldMapRows * kKBlock;
    CUtensorMap tmA;
    const cuuint64_t dims[3] = {(cuuint64_t)kRow, (cuuint64_t)(parts * kTileM / kFoldMapRows), (cuuint64_t)(4 * pairs) * f.kblocks};
    const cuuint64_t strides[2] = {(cuuint64_t)kRow * 2, (cuuint64_t)(parts * kFoldPart)};
    const cuuint32_t box[3] = {(cuuint32_t)kRow, (cuuint32_t)(parts * kTileM / kFoldMapRows), 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    if (!encode_tensor_map(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT16, ring, dims, strides, box, estr,
                           CU_TENSOR_MAP_SWIZZLE_NONE, 3))
        return cudaErrorInvalidValue;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg =
        launch_config(&attr, (unsigned)(2 * pairs), sh.smem, s);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fused_for(mode, chan, rot != nullptr), P, f.tmap2_bhi, f.tmap2_blo, tmA);
    if (facts) *facts = {2 * pairs, 1, 0, rexp ? 2 : 1};       // FP16X3's exponents ran before
    return e;
}
