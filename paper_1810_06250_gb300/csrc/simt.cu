// FP32 CUDA-core RM synthesis with the fused peak map.
//
// The paper's kernel (Sec. 3) gives each thread one Faraday depth and loops
// over channels, computing sin/cos per (channel, phi) in FP32.  Here a block
// owns 256 lines of sight and walks all phi in tiles of 64; per chunk of 16
// channels the 16 x 64 (cos, sin) tile is shared by the block's 256 lines of
// sight, and each thread accumulates an 8 LOS x 8 phi register tile: 64 complex
// MACs = 256 FMAs per channel for 8 shared-memory vector loads, so the FMA pipe,
// not shared-memory bandwidth, sets the rate.  The chunks stream through a
// two-stage cp.async pipeline, so the next chunk's loads overlap this one's FMAs.
//   FLY   : (cos, sin) = sincosf(phi_k * 2(lambda_j^2 - lambda_0^2)) in FP32
//           (the paper's method, argument and reduction in FP32);
//   TABLE : (cos, sin) read from the plan's FP32 table built in FP64.
// On a phi grid symmetric about zero (FOLD) cos is even and sin odd in phi, so
// the four sums Qc, Qs, Uc, Us of a depth phi >= 0 give F at +phi and -phi:
// 4 FMAs per (LOS, channel) for two outputs instead of 8.  The register tile is
// then 8 LOS x 4 pairs, 128 FMAs per channel for 6 vector loads, and the copies
// weigh twice as much: channel-major cubes whose rows start on 16 bytes copy 4 LOS
// at a time.  262,144 LOS x 360 active channels x 401 phi: table 6.82 -> 3.61 ms,
// on the fly 6.97 -> 3.70 ms (rows not aligned 4.58, LOS-major 7.05 -> 4.64 ms).
// The FMAs are packed over two LOS (one instruction, the rounding of two): the issue slots
// were the bound, now the FMA pipe is busy 67 % of the time.  Table 3.56 -> 3.33 ms, on the
// fly 3.66 -> 3.32 ms, rows not aligned 4.53 -> 4.31 ms, LOS-major 4.61 -> 4.40 ms.
// The peak of |F| (Sec. 2.2) is reduced in registers over the block's phi
// tiles, so F never has to be re-read.
#include <cooperative_groups.h>
#include <limits.h>

#include <algorithm>

#include "rms_internal.h"

namespace cg = cooperative_groups;

namespace {

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
constexpr size_t kSimtSmem = 2 * sizeof(Stage);

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
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

__device__ __forceinline__ void load8(const float *p, float2 (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
}

// Each thread copies one channel of every chunk: ISSUE_CH(tid) is that channel's
// slot in the chunk, and its active-channel index is loaded one chunk ahead
// (act), so no global load latency sits in front of the copies.
template <int LAYOUT>
__device__ __forceinline__ int issue_ch(int tid)
{
    return LAYOUT == RMS_CHAN_MAJOR ? tid / (256 / CH) : tid % CH;
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
    if (LAYOUT == RMS_CHAN_MAJOR && a.vec4) {
        // 16 threads per channel, each 4 x 4 LOS (256-byte runs along LOS; nlos is a
        // multiple of 4, so a group of 4 is whole or beyond the end)
#pragma unroll
        for (int r = 0; r < TL / (256 / CH) / 4; ++r) {
            const int m = 4 * (tid % (256 / CH) + r * (256 / CH));
            const bool ok = act >= 0 && l0 + m < a.nlos;
            const int64_t off = ok ? (int64_t)act * a.nlos + l0 + m : 0;
            cp_async<16>(&st.q[c][m], a.Q + off, ok);
            cp_async<16>(&st.u[c][m], a.U + off, ok);
        }
    } else if (LAYOUT == RMS_CHAN_MAJOR) {
        // 16 threads per channel, each 16 LOS at stride 16 (64-byte runs along LOS)
#pragma unroll 4
        for (int r = 0; r < TL / (256 / CH); ++r) {
            const int m = tid % (256 / CH) + r * (256 / CH);
            const bool ok = act >= 0 && l0 + m < a.nlos;
            const int64_t off = ok ? (int64_t)act * a.nlos + l0 + m : 0;
            cp_async<4>(&st.q[c][m], a.Q + off, ok);
            cp_async<4>(&st.u[c][m], a.U + off, ok);
        }
    } else {
        // consecutive threads take consecutive channels of one LOS
#pragma unroll 4
        for (int r = 0; r < TL / (256 / CH); ++r) {
            const int m = tid / CH + r * (256 / CH);
            const bool ok = act >= 0 && l0 + m < a.nlos;
            const int64_t off = ok ? (l0 + m) * a.nchan + act : 0;
            cp_async<4>(&st.q[c][m], a.Q + off, ok);
            cp_async<4>(&st.u[c][m], a.U + off, ok);
        }
    }
    if (!FLY) {
#pragma unroll
        for (int i = tid; i < CH * W; i += 256) {
            const int c = i / W, k = i % W;
            const bool ok = c0 + c < a.nact && p0 + k < a.ncol;
            const int64_t off = ok ? (int64_t)(c0 + c) * a.nphi + a.kplus + p0 + k : 0;
            cp_async<8>(&st.cs[c][k], a.table + off, ok);
        }
    }
}

// on-the-fly phases: the operands of a thread's CH * TP / 256 phase-tile
// entries are loaded one chunk ahead and turned into (w cos, w sin) after the
// current chunk's accumulation, so their load latency is hidden behind it
template <bool FOLD>
struct FlyOps {
    static constexpr int W = FOLD ? TP / 2 : TP, kPer = CH * W / 256;
    float ph[kPer], l2[kPer], w[kPer];
};

template <bool FOLD>
__device__ __forceinline__ void fly_load(const SimtArgs &a, FlyOps<FOLD> &o, int c0, int p0, int tid)
{
#pragma unroll
    for (int r = 0; r < FlyOps<FOLD>::kPer; ++r) {
        const int i = tid + 256 * r, c = i / FlyOps<FOLD>::W, k = i % FlyOps<FOLD>::W;
        const bool ok = c0 + c < a.nact && p0 + k < a.ncol;
        // a padded entry gets weight 0 (and phase 0), hence (0, 0)
        o.ph[r] = ok ? __ldg(a.phi32 + a.kplus + p0 + k) : 0.f;
        o.l2[r] = ok ? __ldg(a.l2x + c0 + c) : 0.f;
        o.w[r] = ok ? __ldg(a.w32 + c0 + c) : 0.f;
    }
}

template <bool FOLD>
__device__ __forceinline__ void fly_store(Stage &st, const FlyOps<FOLD> &o, int tid)
{
#pragma unroll
    for (int r = 0; r < FlyOps<FOLD>::kPer; ++r) {
        const int i = tid + 256 * r, c = i / FlyOps<FOLD>::W, k = i % FlyOps<FOLD>::W;
        float sn, cs;
        sincosf(o.ph[r] * o.l2[r], &sn, &cs);
        st.cs[c][k] = make_float2(o.w[r] * cs, o.w[r] * sn);
    }
}

// Pipeline state carried from one phi tile to the next.
struct Pipe {
    int t;          // (phi tile, channel chunk) pair being accumulated
    int total, nck;
    int32_t act;    // active-channel index for the next copy
    int rank, size; // this block's tiles: rank, rank + size, ... (its place in the cluster)
    __device__ __forceinline__ int chunk(int n) const { return n % nck; }
    __device__ __forceinline__ int tile(int n) const { return rank + (n / nck) * size; }
};

// One phi tile starting at column p0: accumulate all channel chunks, then scale,
// store and update the running peak.  JJ: pairs-of-16 columns of the tile that hold
// grid points (4, folded 2, for a full tile; the last, partial tile drops the columns
// beyond).
template <int JJ, bool FLY, bool FOLD, int LAYOUT>
__device__ __forceinline__ void phi_tile(const SimtArgs &a, Stage *stage, int64_t l0, int p0, Pipe &pp,
                                         FlyOps<FOLD> &fo, float (&bm)[8], int (&bi)[8])
{
    constexpr int NJ = 2 * JJ, W = FOLD ? TP / 2 : TP, NS = FOLD ? 4 : 2;
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    // sums of a (LOS, column): Re, Im of F, or folded Qc, Us, Uc, Qs
    // of LOS 2 i and 2 i + 1: one packed FMA feeds both
    float2 acc[4][NJ][NS];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int x = 0; x < NS; ++x) acc[i][j][x] = make_float2(0.f, 0.f);

    for (int ck = 0; ck < pp.nck; ++ck, ++pp.t) {
        const int n = pp.t + 1;
        if (n < pp.total) {
            issue<FLY, FOLD, LAYOUT>(a, stage[n & 1], l0, pp.chunk(n) * CH, pp.tile(n) * W, pp.act, tid);
            if (FLY) fly_load<FOLD>(a, fo, pp.chunk(n) * CH, pp.tile(n) * W, tid);
            if (n + 1 < pp.total) pp.act = load_active<LAYOUT>(a, pp.chunk(n + 1) * CH, tid);
        }
        cp_commit();
        cp_wait_prev();
        __syncthreads();
        const Stage &st = stage[pp.t & 1];
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
                    float2(&s)[NS] = acc[i][j];
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
        // stage n & 1 was last read before the previous trailing barrier
        if (FLY && n < pp.total) fly_store<FOLD>(stage[n & 1], fo, tid);
        __syncthreads();
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
            float s[NS];
#pragma unroll
            for (int x = 0; x < NS; ++x) s[x] = i & 1 ? acc[i >> 1][j][x].y : acc[i >> 1][j][x].x;
            const int k = a.kplus + col;
            const float fr = (FOLD ? s[0] + s[1] : s[0]) * a.scale;
            const float fi = (FOLD ? s[2] - s[NS - 1] : s[1]) * a.scale;
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

template <bool FLY, bool FOLD, int LAYOUT>
__global__ void __launch_bounds__(256, 1) simt_kernel(const SimtArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float pk_m[TL];
    __shared__ int pk_k[TL];
    Stage *stage = reinterpret_cast<Stage *>(smem_raw);

    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const cg::cluster_group cluster = cg::this_cluster();
    Pipe pp;
    pp.rank = (int)cluster.block_rank();
    pp.size = (int)cluster.num_blocks();
    const int64_t l0 = (int64_t)(blockIdx.x / pp.size) * TL;
    pp.nck = (a.nact + CH - 1) / CH;
    constexpr int W = FOLD ? TP / 2 : TP;
    const int ntiles = (a.ncol + W - 1) / W;        // the cluster has at most as many blocks
    pp.total = pp.nck * ((ntiles - pp.rank + pp.size - 1) / pp.size);
    pp.t = 0;

    float bm[8];
    int bi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { bm[i] = -1.0f; bi[i] = INT_MAX; }

    // two-stage pipeline over (phi tile, channel chunk) pairs t: the copies of
    // pair t + 1 are in flight while pair t is accumulated
    FlyOps<FOLD> fo;
    issue<FLY, FOLD, LAYOUT>(a, stage[0], l0, 0, pp.rank * W, load_active<LAYOUT>(a, 0, tid), tid);
    cp_commit();
    pp.act = pp.total > 1 ? load_active<LAYOUT>(a, pp.chunk(1) * CH, tid) : -1;
    if (FLY) {
        fly_load<FOLD>(a, fo, 0, pp.rank * W, tid);
        fly_store<FOLD>(stage[0], fo, tid);
    }
    const int full = a.ncol / W, rem = a.ncol - full * W;
    int it = pp.rank;
    for (; it < full; it += pp.size) phi_tile<W / 16, FLY, FOLD, LAYOUT>(a, stage, l0, it * W, pp, fo, bm, bi);
    // the last, partial tile computes only the pairs-of-16 that hold grid points
    if (it == full) {
        switch ((rem + 15) / 16) {
        case 1: phi_tile<1, FLY, FOLD, LAYOUT>(a, stage, l0, full * W, pp, fo, bm, bi); break;
        case 2: phi_tile<2, FLY, FOLD, LAYOUT>(a, stage, l0, full * W, pp, fo, bm, bi); break;
        case 3: if constexpr (!FOLD) phi_tile<3, FLY, FOLD, LAYOUT>(a, stage, l0, full * W, pp, fo, bm, bi); break;
        case 4: if constexpr (!FOLD) phi_tile<4, FLY, FOLD, LAYOUT>(a, stage, l0, full * W, pp, fo, bm, bi); break;
        default: break;
        }
    }

    // reduce the peak over the 8 threads (tx) that share each line of sight
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
        if (tx == 0) { pk_m[8 * ty + i] = m; pk_k[8 * ty + i] = k; }
    }
    // the cluster's blocks hold disjoint phi of the same LOS: its first block merges them
    if (pp.size > 1) cluster.sync();
    else __syncthreads();
    if (pp.rank == 0) {
        float m = pk_m[tid];
        int k = pk_k[tid];
        for (int r = 1; r < pp.size; ++r) {
            const float mo = cluster.map_shared_rank(pk_m, r)[tid];
            const int ko = cluster.map_shared_rank(pk_k, r)[tid];
            if (better(mo, ko, m, k)) { m = mo; k = ko; }
        }
        const int64_t l = l0 + tid;
        if (l < a.nlos) {
            const bool ok = k != INT_MAX;
            if (a.pidx) a.pidx[l] = ok ? k : -1;
            if (a.pabs) a.pabs[l] = ok ? sqrtf(m) : __int_as_float(0x7fc00000);
            if (a.pphi) a.pphi[l] = ok ? a.phi32[k] : __int_as_float(0x7fc00000);
        }
    }
    if (pp.size > 1) cluster.sync();    // no block leaves while another reads its shared memory
}

cudaLaunchConfig_t launch_config(cudaLaunchAttribute *attr, unsigned grid, unsigned cluster, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(TL);
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
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSimtSmem);
        for (int c = 1; c <= 8 && e == cudaSuccess; ++c) {
            cudaLaunchAttribute attr;
            const cudaLaunchConfig_t cfg = launch_config(&attr, (unsigned)(c * p->num_sms), (unsigned)c, 0);
            int n = 0;
            e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
            p->simt_clusters[c - 1] = layout == RMS_CHAN_MAJOR ? n : std::min(n, p->simt_clusters[c - 1]);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
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
    const bool fold = p.fold.on;
    a.ncol = fold ? p.fold.ncol : p.nphi;
    a.kplus = fold ? p.fold.kplus : 0;
    a.kminus = p.fold.kminus;
    a.vec4 = nlos % 4 == 0 && !((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(U)) & 15);
    const int64_t blocks = (nlos + TL - 1) / TL;
    // One block fits an SM, and its phi tiles re-read the block's data anyway, so a
    // cluster of up to 8 blocks shares out the phi tiles of 256 LOS where that needs
    // fewer rounds of tiles over the device (the smallest such cluster).  401 phi x 360
    // channels: 3,000 LOS 522 -> 84 us, 10,000 LOS 520 -> 207, 100,000 unchanged (1.53 ms).
    const int width = fold ? TP / 2 : TP, ntiles = (a.ncol + width - 1) / width;
    int64_t best = INT64_MAX;
    unsigned cluster = 1;
    for (int c = 1; c <= std::min(8, ntiles); ++c) {
        if (p.simt_clusters[c - 1] < 1) continue;
        const int64_t rounds = (blocks + p.simt_clusters[c - 1] - 1) / p.simt_clusters[c - 1] * ((ntiles + c - 1) / c);
        if (rounds < best) { best = rounds; cluster = (unsigned)c; }
    }
    if (blocks * cluster > 0x7fffffff) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(&attr, (unsigned)blocks * cluster, cluster, s);
    return cudaLaunchKernelEx(&cfg, kernel_of(fly, fold, layout), a);
}
