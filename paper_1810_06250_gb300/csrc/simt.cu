// FP32 CUDA-core RM synthesis with the fused peak map.
//
// The paper's kernel (Sec. 3) gives each thread one Faraday depth and loops
// over channels, computing sin/cos per (channel, phi) in FP32.  Here a block
// owns 256 lines of sight and walks all phi in tiles of 64; per chunk of 16
// channels the 16 x 64 (cos, sin) tile is shared by the block's 256 lines of
// sight, and each thread accumulates an 8 LOS x 8 phi register tile: 64 complex
// MACs = 256 FMAs per channel for 8 shared-memory vector loads, so the FMA pipe,
// not shared-memory bandwidth, sets the rate.  Four copying warps stream the chunks
// through a four-stage cp.async pipeline for the eight accumulating ones, which meet
// no barrier of the block while they run.  (With every warp copying between two barriers a
// chunk, a third of the time had no FMA in flight: 262,144 LOS x 360 active channels x 401
// phi folded, below, table 3.33 -> 2.75 ms, on the fly 3.32 -> 2.85, LOS-major 4.40 -> 3.28.)
//   FLY   : (cos, sin) = sincosf(phi_k * 2(lambda_j^2 - lambda_0^2)) in FP32
//           (the paper's method, argument and reduction in FP32);
//   TABLE : (cos, sin) read from the plan's FP32 table built in FP64.
// On a phi grid symmetric about zero (FOLD) cos is even and sin odd in phi, so
// the four sums Qc, Qs, Uc, Us of a depth phi >= 0 give F at +phi and -phi:
// 4 FMAs per (LOS, channel) for two outputs instead of 8.  The register tile is
// then 8 LOS x 4 pairs, 128 FMAs per channel for 6 vector loads, and the copies
// weigh twice as much: channel-major cubes whose rows start on 16 bytes copy 4 LOS
// at a time.  Folding took the table path from 6.82 to 3.61 ms, LOS-major from 7.05 to 4.64.
// The FMAs are packed over two LOS (one instruction, the rounding of two), which freed the
// issue slots that bound them: table 3.56 -> 3.33 ms, LOS-major 4.61 -> 4.40 ms.
// The peak of |F| (Sec. 2.2) is reduced in registers over the block's phi
// tiles, so F never has to be re-read.
#include <cooperative_groups.h>
#include <limits.h>

#include <algorithm>
#include <type_traits>

#include "rms_internal.h"

namespace cg = cooperative_groups;

namespace {

#include "tc_ptx.cuh"

constexpr int TL = 256;   // lines of sight per block (32 thread rows x 8)
constexpr int TP = 64;    // phi per tile (8 thread columns x 8, as 4 pairs at stride 16);
                          // folded: 32 phi columns, each a +-phi pair (8 thread columns x 4)
constexpr int CH = 16;    // channels per chunk
constexpr int LDQ = TL + 4;

// one pipeline stage in shared memory: the chunk's data and phase tiles
struct Stage {
    float q[CH][LDQ];
    float u[CH][LDQ];
    float2 cs[CH][TP];     // (w cos, w sin)
};
constexpr int NS = 4;      // stages
constexpr int NP = 128;    // copying threads
constexpr int kThreads = TL + NP;
constexpr size_t kSimtSmem = NS * sizeof(Stage);
// registers a thread: the launch's share, and after the split (256 x 232 + 128 x 40 = 384 x 168)
constexpr int kRegsLaunch = 168, kRegsSum = 232, kRegsCopy = 40;
static_assert(TL * kRegsSum + NP * kRegsCopy <= kThreads * kRegsLaunch, "register split");
constexpr int64_t kWaitNs = 20000000000;    // no wait of a block on itself comes near this

struct SimtArgs {
    const float *Q, *U;
    int64_t nlos;
    int32_t nchan, nact, nphi;
    const int32_t *active;
    const float *l2x;      // [nact] 2 (lambda^2 - lambda_0^2), FP32
    const float *w32;      // [nact]
    const float *phi32;    // [nphi]
    const float2 *table;   // [nact][nphi]
    float scale;           // K
    int32_t ncol;          // phi columns: nphi, or folded the ceil(nphi / 2) depths phi >= 0
    int32_t kplus, kminus; // column i is sample kplus + i (folded: and kminus - i)
    int32_t vec4;          // channel-major rows start on 16 bytes: 4 LOS per copy
    float *F;
    int32_t *pidx;
    float *pabs, *pphi;
    int *err;
    // balanced form (one CTA per SM): the cost of a block's phi tiles, in 16-column pieces, and
    // what two CTAs that share a block exchange: [CTA][2][TL] peaks, [CTA] arrivals (0 at launch)
    int32_t balanced, block_cost;
    int64_t blocks;
    float *part_m;
    int32_t *part_k;
    int32_t *arrived;
};

__device__ __forceinline__ bool better(float m, int i, float bm, int bi)
{
    return m > bm || (m == bm && i < bi);
}

// asynchronous global -> shared copy of 4, 8 or 16 bytes; a false predicate
// writes zeros and reads nothing (the source is then any valid address)
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src, bool ok)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES),
                 "r"(ok ? BYTES : 0)
                 : "memory");
}
// arrive on an mbarrier once this thread's copies so far have landed
__device__ __forceinline__ void cp_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void load8(const float *p, float2 (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
}

// Each copying thread takes one channel of every chunk: ISSUE_CH(tid) is that channel's
// slot in the chunk, and its active-channel index is loaded one chunk ahead
// (act), so no global load latency sits in front of the copies.
template <int LAYOUT>
__device__ __forceinline__ int issue_ch(int tid)
{
    return LAYOUT == RMS_CHAN_MAJOR ? tid / (NP / CH) : tid % CH;
}

template <int LAYOUT>
__device__ __forceinline__ int32_t load_active(const SimtArgs &a, int c0, int tid)
{
    const int c = c0 + issue_ch<LAYOUT>(tid);
    return c < a.nact ? __ldg(a.active + c) : -1;
}

// fill stage st with channel chunk c0 and phi tile p0 of the block's lines of sight
template <bool FLY, bool FOLD, int LAYOUT>
__device__ __forceinline__ void issue(const SimtArgs &a, Stage &st, int64_t l0, int c0, int p0, int32_t act,
                                      int tid)
{
    const int c = issue_ch<LAYOUT>(tid);
    constexpr int W = FOLD ? TP / 2 : TP;
    constexpr bool chan = LAYOUT == RMS_CHAN_MAJOR;
    // channel-major: 8 threads per channel, each 8 x 4 LOS (128-byte runs along LOS; with vec4
    // nlos is a multiple of 4, so a group of 4 is whole or beyond the end) or 32 LOS at stride
    // 8; LOS-major: consecutive threads take consecutive channels of a LOS, each 32 LOS at
    // stride 8.  The block's last LOS, and channels beyond the last, are zeros.
    const int per = chan && a.vec4 ? 4 : 1, m0 = per * (chan ? tid % (NP / CH) : tid / CH), dm = per * (NP / CH);
    const int64_t step = (int64_t)dm * (chan ? 1 : a.nchan);
    const int n = (int)min((int64_t)TL, a.nlos - l0);
    const int64_t off = chan ? (int64_t)max(act, 0) * a.nlos + l0 + m0 : (l0 + m0) * a.nchan + max(act, 0);
    const float *q = a.Q + off, *u = a.U + off;
    float *dq = &st.q[c][m0], *du = &st.u[c][m0];
    auto copy = [&](auto bytes) {
        constexpr int B = decltype(bytes)::value, steps = TL * (int)sizeof(float) / ((NP / CH) * B);
        if (n == TL) {
#pragma unroll 8
            for (int r = 0; r < steps; ++r) {
                cp_async<B>(dq + r * dm, q, act >= 0);
                cp_async<B>(du + r * dm, u, act >= 0);
                q += step;
                u += step;
            }
        } else {
#pragma unroll 1
            for (int r = 0; r < steps; ++r) {
                const bool ok = act >= 0 && m0 + r * dm < n;
                cp_async<B>(dq + r * dm, ok ? q + r * step : a.Q, ok);
                cp_async<B>(du + r * dm, ok ? u + r * step : a.U, ok);
            }
        }
    };
    if (chan && a.vec4) copy(std::integral_constant<int, 16>());
    else copy(std::integral_constant<int, 4>());
    if (!FLY) {
#pragma unroll
        for (int i = tid; i < CH * W; i += NP) {
            const int c = i / W, k = i % W;
            const bool ok = c0 + c < a.nact && p0 + k < a.ncol;
            const int64_t off = ok ? (int64_t)(c0 + c) * a.nphi + a.kplus + p0 + k : 0;
            cp_async<8>(&st.cs[c][k], a.table + off, ok);
        }
    }
}

// on-the-fly phases: the chunk's (w cos, w sin)
template <bool FOLD>
__device__ __forceinline__ void fly_store(const SimtArgs &a, Stage &st, int c0, int p0, int tid)
{
    constexpr int W = FOLD ? TP / 2 : TP;
#pragma unroll 1
    for (int i = tid; i < CH * W; i += NP) {
        const int c = i / W, k = i % W;
        const bool ok = c0 + c < a.nact && p0 + k < a.ncol;
        // a padded entry gets weight 0 (and phase 0), hence (0, 0)
        const float ph = ok ? __ldg(a.phi32 + a.kplus + p0 + k) : 0.f;
        const float l2 = ok ? __ldg(a.l2x + c0 + c) : 0.f;
        const float w = ok ? __ldg(a.w32 + c0 + c) : 0.f;
        float sn, cs;
        sincosf(ph * l2, &sn, &cs);
        st.cs[c][k] = make_float2(w * cs, w * sn);
    }
}

// Pipeline state: the stage and the parity of its current use, and this block's phi tiles
// rank, rank + size, ... (its place in the cluster).
struct Pipe {
    uint64_t *full, *empty;
    volatile int *abort_flag;
    int s;
    uint32_t ph;
    int nck, rank, size;
    __device__ __forceinline__ void next()
    {
        if (++s == NS) { s = 0; ph ^= 1; }
    }
};

// One phi tile starting at column p0: accumulate all channel chunks, then scale,
// store and update the running peak.  JJ: pairs-of-16 columns of the tile that hold
// grid points (4, folded 2, for a full tile; the last, partial tile drops the columns
// beyond).
template <int JJ, bool FOLD>
__device__ __forceinline__ void phi_tile(const SimtArgs &a, const Stage *stage, int64_t l0, int p0, Pipe &pp,
                                         float (&bm)[8], int (&bi)[8])
{
    constexpr int NJ = 2 * JJ, SUMS = FOLD ? 4 : 2;
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    // sums of a (LOS, column): Re, Im of F, or folded Qc, Us, Uc, Qs
    // of LOS 2 i and 2 i + 1: one packed FMA feeds both
    float2 acc[4][NJ][SUMS];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int x = 0; x < SUMS; ++x) acc[i][j][x] = make_float2(0.f, 0.f);

    for (int ck = 0; ck < pp.nck; ++ck, pp.next()) {
        if (!warp_wait(smem_u32(&pp.full[pp.s]), pp.ph, pp.abort_flag, a.err, kWaitNs)) return;
        const Stage &st = stage[pp.s];
#pragma unroll 2
        for (int c = 0; c < CH; ++c) {
            float2 qv[4], uv[4];
            float cv[NJ], sv[NJ];
            load8(&st.q[c][8 * ty], qv);
            load8(&st.u[c][8 * ty], uv);
            // thread tx owns phi pairs 16 jj + 2 tx + {0, 1}: the 8 threads of a
            // row read 128 contiguous bytes per vector load (no bank conflict)
#pragma unroll
            for (int j = 0; j < NJ; j += 2) {
                const float4 v = *reinterpret_cast<const float4 *>(&st.cs[c][8 * j + 2 * tx]);
                cv[j] = v.x; sv[j] = v.y; cv[j + 1] = v.z; sv[j + 1] = v.w;
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const float2 c2 = make_float2(cv[j], cv[j]), s2 = make_float2(sv[j], sv[j]);
                const float2 n2 = make_float2(-sv[j], -sv[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2(&s)[SUMS] = acc[i][j];
                    // (q + iu)(c - is): Re += q c + u s, Im += u c - q s  (Eqs. qPhi, uPhi)
                    if constexpr (FOLD) {
                        s[0] = __ffma2_rn(qv[i], c2, s[0]);
                        s[1] = __ffma2_rn(uv[i], s2, s[1]);
                        s[2] = __ffma2_rn(uv[i], c2, s[2]);
                        s[3] = __ffma2_rn(qv[i], s2, s[3]);
                    } else {
                        s[0] = __ffma2_rn(qv[i], c2, s[0]);
                        s[0] = __ffma2_rn(uv[i], s2, s[0]);
                        s[1] = __ffma2_rn(uv[i], c2, s[1]);
                        s[1] = __ffma2_rn(qv[i], n2, s[1]);
                    }
                }
            }
        }
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(smem_u32(&pp.empty[pp.s]));
    }

    // epilogue for this phi tile: scale by K, store, update the running peak (lowest
    // index among equals: a +phi sample is above, a folded -phi one below all before it)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t l = l0 + 8 * ty + i;
        float2 *row = reinterpret_cast<float2 *>(a.F) + l * a.nphi;
        const bool st = a.F != nullptr && l < a.nlos;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int col = p0 + 16 * (j >> 1) + 2 * tx + (j & 1);
            if (col >= a.ncol) continue;
            float s[SUMS];
#pragma unroll
            for (int x = 0; x < SUMS; ++x) s[x] = i & 1 ? acc[i >> 1][j][x].y : acc[i >> 1][j][x].x;
            const int k = a.kplus + col;
            const float fr = (FOLD ? s[0] + s[1] : s[0]) * a.scale;
            const float fi = (FOLD ? s[2] - s[SUMS - 1] : s[1]) * a.scale;
            const float m2 = __fadd_rn(__fmul_rn(fr, fr), __fmul_rn(fi, fi));
            if (m2 > bm[i]) { bm[i] = m2; bi[i] = k; }
            if (st) row[k] = make_float2(fr, fi);
            if constexpr (FOLD) {
                const int kn = a.kminus - col;
                if (kn == k) continue;          // phi = 0 is its own partner
                const float gr = (s[0] - s[1]) * a.scale, gi = (s[2] + s[3]) * a.scale;
                const float g2 = __fadd_rn(__fmul_rn(gr, gr), __fmul_rn(gi, gi));
                if (g2 >= bm[i]) { bm[i] = g2; bi[i] = kn; }
                if (st) row[kn] = make_float2(gr, gi);
            }
        }
    }
}

__device__ __forceinline__ void write_peak(const SimtArgs &a, int64_t l, float m, int k)
{
    if (l >= a.nlos) return;
    const bool ok = k != INT_MAX;
    if (a.pidx) a.pidx[l] = ok ? k : -1;
    if (a.pabs) a.pabs[l] = ok ? sqrtf(m) : __int_as_float(0x7fc00000);
    if (a.pphi) a.pphi[l] = ok ? a.phi32[k] : __int_as_float(0x7fc00000);
}

// the accumulating warps
__device__ __forceinline__ void sum_sync() { asm volatile("bar.sync 1, %0;" ::"n"(TL) : "memory"); }

template <bool FLY, bool FOLD, int LAYOUT>
__global__ void __launch_bounds__(kThreads, 1) simt_kernel(const SimtArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float pk_m[2 * TL];
    __shared__ int pk_k[2 * TL];
    __shared__ int second;
    Stage *stage = reinterpret_cast<Stage *>(smem_raw);

    __shared__ uint64_t bars[2 * NS];
    __shared__ int aborted;

    const int tid = threadIdx.x;
    const cg::cluster_group cluster = cg::this_cluster();
    Pipe pp;
    pp.full = bars;
    pp.empty = bars + NS;
    pp.abort_flag = &aborted;
    pp.rank = (int)cluster.block_rank();
    pp.size = (int)cluster.num_blocks();
    pp.nck = (a.nact + CH - 1) / CH;
    pp.s = 0;
    constexpr int W = FOLD ? TP / 2 : TP;
    const int ntiles = (a.ncol + W - 1) / W;        // the cluster has at most as many blocks
    if (tid == 0) {
        aborted = 0;
        for (int i = 0; i < NS; ++i) {
            mbar_init(smem_u32(&pp.full[i]), 2 * NP);     // each copying thread: its copies, and itself
            mbar_init(smem_u32(&pp.empty[i]), TL / 32);
        }
    }
    __syncthreads();

    // This CTA's share: phi tiles t0, t0 + size, .. of one block; or balanced, the run of
    // (block, tile) units whose costs start in its part of the total.
    const int piece = W / 16;
    int64_t b0 = blockIdx.x / pp.size, b1 = b0;        // first and last block
    int t0 = pp.rank, t1 = ntiles;                      // first tile of b0, end of b1's tiles
    if (a.balanced) {
        auto bound = [&](int64_t i, int64_t &b, int &t) {
            const int64_t c = (i * a.blocks * a.block_cost + gridDim.x - 1) / gridDim.x;
            b = c / a.block_cost;
            t = (int)(c - b * a.block_cost + piece - 1) / piece;
            if (t == ntiles) { t = 0; ++b; }
        };
        bound(blockIdx.x, b0, t0);
        bound(blockIdx.x + 1, b1, t1);
        if (t1 == 0) { t1 = ntiles; --b1; }
    }

    if (tid >= TL) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCopy));
        const int t = tid - TL;
        pp.ph = 1;                                  // every stage starts empty
        bool ok = true;
        int32_t act = load_active<LAYOUT>(a, 0, t);
        for (int64_t b = b0; b <= b1 && ok; ++b) {
            const int end = b == b1 ? t1 : ntiles;
            for (int it = b == b0 ? t0 : 0; it < end && ok; it += pp.size)
                for (int ck = 0; ck < pp.nck; ++ck, pp.next()) {
                    ok = wait_bounded(smem_u32(&pp.empty[pp.s]), pp.ph, pp.abort_flag, a.err, kWaitNs);
                    if (!ok) break;
                    issue<FLY, FOLD, LAYOUT>(a, stage[pp.s], b * TL, ck * CH, it * W, act, t);
                    act = load_active<LAYOUT>(a, ck + 1 < pp.nck ? (ck + 1) * CH : 0, t);
                    if (FLY) fly_store<FOLD>(a, stage[pp.s], ck * CH, it * W, t);
                    cp_arrive(smem_u32(&pp.full[pp.s]));
                    mbar_arrive(smem_u32(&pp.full[pp.s]));
                }
        }
        cp_wait_all();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSum));
        pp.ph = 0;
        const int full = a.ncol / W, rem = a.ncol - full * W;
        for (int64_t b = b0; b <= b1; ++b) {
            const int64_t l0 = b * TL;
            const int first = b == b0 ? t0 : 0, end = b == b1 ? t1 : ntiles;
            float bm[8];
            int bi[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { bm[i] = -1.0f; bi[i] = INT_MAX; }
            int it = first;
            for (; it < min(full, end); it += pp.size) phi_tile<W / 16, FOLD>(a, stage, l0, it * W, pp, bm, bi);
            // the last, partial tile computes only the pairs-of-16 that hold grid points
            if (it == full && it < end) {
                switch ((rem + 15) / 16) {
                case 1: phi_tile<1, FOLD>(a, stage, l0, full * W, pp, bm, bi); break;
                case 2: phi_tile<2, FOLD>(a, stage, l0, full * W, pp, bm, bi); break;
                case 3: if constexpr (!FOLD) phi_tile<3, FOLD>(a, stage, l0, full * W, pp, bm, bi); break;
                case 4: if constexpr (!FOLD) phi_tile<4, FOLD>(a, stage, l0, full * W, pp, bm, bi); break;
                default: break;
                }
            }
            // reduce the peak over the 8 threads (tx) that share each line of sight
            const int tx = tid & 7, ty = tid >> 3;
            float *const pm = pk_m + (b & 1) * TL;
            int *const pk = pk_k + (b & 1) * TL;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float m = bm[i];
                int k = bi[i];
#pragma unroll
                for (int off = 4; off >= 1; off >>= 1) {
                    const float mo = __shfl_xor_sync(0xffffffffu, m, off);
                    const int ko = __shfl_xor_sync(0xffffffffu, k, off);
                    if (better(mo, ko, m, k)) { m = mo; k = ko; }
                }
                if (tx == 0) { pm[8 * ty + i] = m; pk[8 * ty + i] = k; }
            }
            if (!a.balanced) break;
            sum_sync();
            float m = pm[tid];
            int k = pk[tid];
            bool mine = true;
            if (first > 0 || end < ntiles) {
                // the block's other tiles are the neighbour CTA's: whoever comes second merges
                const int64_t slot = blockIdx.x - (first > 0 ? 1 : 0);
                const int side = first > 0;
                a.part_m[(2 * slot + side) * TL + tid] = m;
                a.part_k[(2 * slot + side) * TL + tid] = k;
                __threadfence();
                sum_sync();
                if (tid == 0) second = atomicAdd(a.arrived + slot, 1);
                sum_sync();
                mine = second != 0;
                if (mine) {
                    __threadfence();
                    const float mo = __ldcg(a.part_m + (2 * slot + 1 - side) * TL + tid);
                    const int ko = __ldcg(a.part_k + (2 * slot + 1 - side) * TL + tid);
                    if (better(mo, ko, m, k)) { m = mo; k = ko; }
                }
            }
            if (mine) write_peak(a, l0 + tid, m, k);
        }
    }
    if (a.balanced) return;
    // the cluster's blocks hold disjoint phi of the same LOS: its first block merges them
    float *const pm = pk_m + (b0 & 1) * TL;
    int *const pk = pk_k + (b0 & 1) * TL;
    if (pp.size > 1) cluster.sync();
    else __syncthreads();
    if (pp.rank == 0 && tid < TL) {
        float m = pm[tid];
        int k = pk[tid];
        for (int r = 1; r < pp.size; ++r) {
            const float mo = cluster.map_shared_rank(pm, r)[tid];
            const int ko = cluster.map_shared_rank(pk, r)[tid];
            if (better(mo, ko, m, k)) { m = mo; k = ko; }
        }
        write_peak(a, b0 * TL + tid, m, k);
    }
    if (pp.size > 1) cluster.sync();    // no block leaves while another reads its shared memory
}

cudaLaunchConfig_t launch_config(cudaLaunchAttribute *attr, unsigned grid, unsigned cluster, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSimtSmem;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cluster;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

using SimtKernel = void (*)(SimtArgs);
SimtKernel kernel_of(bool fly, bool fold, int layout)
{
    const bool chan = layout == RMS_CHAN_MAJOR;
    if (fly) {
        if (fold) return chan ? simt_kernel<true, true, RMS_CHAN_MAJOR> : simt_kernel<true, true, RMS_LOS_MAJOR>;
        return chan ? simt_kernel<true, false, RMS_CHAN_MAJOR> : simt_kernel<true, false, RMS_LOS_MAJOR>;
    }
    if (fold) return chan ? simt_kernel<false, true, RMS_CHAN_MAJOR> : simt_kernel<false, true, RMS_LOS_MAJOR>;
    return chan ? simt_kernel<false, false, RMS_CHAN_MAJOR> : simt_kernel<false, false, RMS_LOS_MAJOR>;
}

}  // namespace

// Clusters of 1 .. 8 blocks that the device holds at once (a cluster lives inside one
// GPC, so sizes that do not divide a GPC's SMs leave some idle).
cudaError_t simt_prepare(rms_plan_s *p)
{
    const bool fly = p->precision == RMS_FP32_SIMT_FLY;
    for (int layout : {RMS_CHAN_MAJOR, RMS_LOS_MAJOR}) {
        const SimtKernel kern = kernel_of(fly, p->fold.on, layout);
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, kern);
        if (e == cudaSuccess && fa.numRegs != kRegsLaunch) e = cudaErrorInvalidConfiguration;    // the split counts on it
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSimtSmem);
        for (int c = 1; c <= 8 && e == cudaSuccess; ++c) {
            cudaLaunchAttribute attr;
            const cudaLaunchConfig_t cfg = launch_config(&attr, (unsigned)(c * p->num_sms), (unsigned)c, 0);
            int n = 0;
            e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
            p->simt_clusters[c - 1] = layout == RMS_CHAN_MAJOR ? n : std::min(n, p->simt_clusters[c - 1]);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaMalloc(reinterpret_cast<void **>(&p->d_simt_part), ((size_t)4 * TL + 1) * p->num_sms * sizeof(float));
}

cudaError_t launch_simt(const rms_plan_s &p, bool fly, const float *Q, const float *U, int64_t nlos,
                        int layout, float *F, int32_t *pidx, float *pabs, float *pphi,
                        cudaStream_t s)
{
    SimtArgs a;
    a.Q = Q;
    a.U = U;
    a.nlos = nlos;
    a.nchan = p.nchan;
    a.nact = p.nact;
    a.nphi = p.nphi;
    a.active = p.d_active;
    a.l2x = p.d_l2x32;
    a.w32 = p.d_w32;
    a.phi32 = p.d_phi32;
    a.table = p.d_table;
    a.scale = (float)p.K;
    a.F = F;
    a.pidx = pidx;
    a.pabs = pabs;
    a.pphi = pphi;
    a.err = p.d_err;
    const bool fold = p.fold.on;
    a.ncol = fold ? p.fold.ncol : p.nphi;
    a.kplus = fold ? p.fold.kplus : 0;
    a.kminus = p.fold.kminus;
    a.vec4 = nlos % 4 == 0 && !((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(U)) & 15);
    const int64_t blocks = (nlos + TL - 1) / TL;
    // One block fits an SM, and its phi tiles re-read the block's data anyway, so a
    // cluster of up to 8 blocks shares out the phi tiles of 256 LOS where that needs
    // fewer rounds of tiles over the device (the smallest such cluster).  401 phi x 360
    // channels: 3,000 LOS 522 -> 84 us, 10,000 LOS 520 -> 207 (before the copying warps;
    // now 68 and 162 us).
    const int width = fold ? TP / 2 : TP, ntiles = (a.ncol + width - 1) / width;
    unsigned cluster = 1;
    int64_t grid = blocks;
    // More blocks than SMs: one CTA per SM takes an equal run of all blocks' phi tiles, where whole blocks
    // in rounds would leave the last round partly empty; a run's first and last block may be shared with
    // the neighbour CTA, whose peaks are merged by the later of the two.  401 phi x 360 channels: 60,000
    // LOS (1.5 blocks per SM) 793 -> 674 us, 100,000 (2.6) 1,185 -> 1,066, 262,144 (6.7) 2.75 -> 2.68 ms.
    a.balanced = blocks > p.num_sms;
    a.blocks = blocks;
    a.block_cost = a.ncol / width * (width / 16) + (a.ncol % width + 15) / 16;
    if (a.balanced) {
        grid = p.num_sms;
        const size_t n = (size_t)2 * p.num_sms * TL;
        a.part_m = p.d_simt_part;
        a.part_k = reinterpret_cast<int32_t *>(p.d_simt_part + n);
        a.arrived = a.part_k + n;
        const cudaError_t e = cudaMemsetAsync(a.arrived, 0, p.num_sms * sizeof(int32_t), s);
        if (e != cudaSuccess) return e;
    } else {
        int64_t best = INT64_MAX;
        for (int c = 1; c <= std::min(8, ntiles); ++c) {
            if (p.simt_clusters[c - 1] < 1) continue;
            const int64_t rounds = (blocks + p.simt_clusters[c - 1] - 1) / p.simt_clusters[c - 1] * ((ntiles + c - 1) / c);
            if (rounds < best) { best = rounds; cluster = (unsigned)c; }
        }
        grid = blocks * cluster;
    }
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(&attr, (unsigned)grid, cluster, s);
    return cudaLaunchKernelEx(&cfg, kernel_of(fly, fold, layout), a);
}
