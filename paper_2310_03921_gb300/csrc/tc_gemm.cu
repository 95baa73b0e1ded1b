// Split-precision BF16 GEMM on the sm_103a tensor cores (tcgen05 + TMA + TMEM).
//
//   C[r][c] = sum_k (Ahi Bhi + Ahi Blo + Alo Bhi)[r][c][k]
//
// A and B are K-major BF16 ([rows][K] and [cols][K]); hi + lo represent an FP32
// value to ~16 significant bits, so the three products recover an FP32-grade
// dot product with FP32 accumulation in TMEM (the lo*lo term is below the
// FP32 accumulation error).  One 128 x BN output tile per CTA:
//   warp 0       TMA producer (one lane) over K blocks of 64, STAGES-deep ring
//   warp 1       TMEM allocation and MMA issue (one lane), tcgen05.commit to
//                free ring slots and to signal the accumulator
//   warps 2..9   epilogue: tcgen05.ld of TMEM lanes (two warps per lane
//                quadrant, one column half each)
// Every mbarrier wait is bounded by wall time; on expiry the CTA records an
// error code in *err, stops issuing work, and still releases its TMEM.
//
// Epilogues:
//   EPI_KERNEL   the sparse-GP kernel of Eqs. 2 and 13 on centred operands:
//                q = C + s_col + t_row, W = zeta delta^2 alpha q^(zeta-1) stored as
//                BF16 hi/lo, per-tile partial sums of delta^2 alpha q^zeta (taken
//                as W q, divided by zeta at the end) and of W.  Its epilogue
//                bounds it, in instructions and stores: a lane owns a row, so
//                direct stores touch 32 lines 16 bytes at a time.  Each warp
//                stages 32 x 32 blocks of W in shared memory and stores them by
//                TMA, which also clips the last rows; zeta = 4 (every workload's)
//                has its power written out, 14 instructions per element with
//                it where the general loop and direct stores took 33.  A step
//                of 32768 atoms 1444 -> 1316 us, of 110592 atoms 9059 -> 8144
//                us, 512 four-species boxes 4059 -> 3843 us.
//   EPI_QPOW     per atom and sparse point, W' = zeta delta^2 q^(zeta-1) and
//                delta^2 q^zeta (FP32) for the K_NM rows, bound by its 8 bytes
//                per element, stored the same way (K_NM of 200 silicon cells
//                7020 -> 6891 us)
//   EPI_STORE    FP32 store of C
#include <cuda.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "gap_internal.h"
#include "tc_gemm.h"
#include "tc_prim.cuh"

namespace {

using namespace tcp;

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kEpiWarps = 8;

struct SharedTail {
    uint64_t full[4];
    uint64_t empty[4];
    uint64_t acc_full[2];    // MMA -> epilogue, per TMEM accumulator buffer
    uint64_t acc_empty[2];   // epilogue -> MMA (every epilogue warp arrives)
    uint64_t mma_done;       // the issuer's last MMA
    uint32_t tmem_base;
    int abort;
};

// A warp's staging of one W plane: 32 rows of 32 BF16, 64-byte swizzle.
constexpr uint32_t kStagePlane = 32 * 64;

// q^e for 0 <= e < 64 by square-and-multiply over the six bits of e: fully
// unrolled (e is the same for every thread), so the epilogue's element loops
// keep no data-dependent inner loop.
__device__ __forceinline__ float powi_small(float q, int e)
{
    float r = 1.f, b = q;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        if ((e >> k) & 1) r *= b;
        b *= b;
    }
    return r;
}

// One GEMM problem of a launch: its operand maps (A hi / mid-or-lo / lo, B
// the same), sizes, first tile in the launch's tile order, and epilogue.
struct TcProblem {
    CUtensorMap mA[3], mB[3], mW[3];  // mW (stores): EPI_KERNEL's W planes, EPI_QPOW's W' and k
    int rows, cols, K, tile0;
    int kpart, tiles_part;  // K blocks per part of K, tiles of one part
    TcEpilogue ep;
};
// G problems in one persistent launch (the GEMMs of a batch's GPs): tiles
// are numbered problem after problem.
template <int G> struct TcProblems {
    int n, n_tiles;
    TcProblem p[G];
};

// NS = number of BF16 planes per operand: 2 (hi, lo: three MMAs per K step)
// or 3 (hi, mid, lo: the six products with plane-index sum <= 2, an
// FP32-grade product).
// EW = epilogue warps: 8 (two column groups), or 12 (three, on 192-column
// tiles).
template <int BN, int STAGES, int EPI, int NS, int G, int EW>
__global__ void __launch_bounds__(32 * (2 + EW), 1)
k_tc_gemm(const __grid_constant__ TcProblems<G> P, int *err)
{
    static_assert(BN == 128 || BN == 192 || BN == 256, "tile width");
    static_assert(NS == 2 || NS == 3, "planes");
    static_assert(EW == 8 || (EW == 12 && (EPI == EPI_KERNEL || EPI == EPI_STORE) && BN == 192), "epilogue warps");
    constexpr int kThreads = 32 * (2 + EW);  // this instantiation's block
    constexpr int NG = EW / 4;               // epilogue column groups
    constexpr uint32_t TMEM_COLS = 2 * BN <= 256 ? 256 : 512;  // two accumulators, a power of two
    constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
    constexpr uint32_t STAGE_BYTES = NS * A_BYTES + NS * B_BYTES;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    // after the ring (which keeps filling for the next tile while an epilogue
    // runs): the epilogue warps' store staging, the barriers, per-column constants
    constexpr uint32_t STAGING = EPI != EPI_STORE ? EW * 2 * kStagePlane : 0;
    unsigned char *staging = smem + STAGES * STAGE_BYTES;
    SharedTail *tail = reinterpret_cast<SharedTail *>(staging + STAGING);
    unsigned char *scratch = staging + STAGING + ((sizeof(SharedTail) + 127) & ~size_t(127));
    float *col_s = reinterpret_cast<float *>(scratch), *col_a = col_s + BN;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Persistent: CTA b takes tiles b, b + gridDim.x, ... (row tile major, so
    // the CTAs running at one time share A row tiles in L2).  The TMA ring
    // and the two TMEM accumulators continue across tiles, so the epilogue of
    // one tile overlaps the loads and MMAs of the next.
    const int n_tiles = P.n_tiles;
    // tile -> (problem, tile within it, K blocks [kb0, kb1) of its part of K);
    // returns the part
    auto locate = [&](int tile, int &gi, int &lt, int &kb0, int &kb1) {
        gi = 0;
#pragma unroll
        for (int q = 1; q < G; ++q)
            if (q < P.n && tile >= P.p[q].tile0) gi = q;
        lt = tile - P.p[gi].tile0;
        const int kblocks = (P.p[gi].K + BK - 1) / BK;
        if (EPI != EPI_STORE) {
            kb0 = 0;
            kb1 = kblocks;
            return 0;
        }
        const int part = lt / P.p[gi].tiles_part;
        lt -= part * P.p[gi].tiles_part;
        kb0 = part * P.p[gi].kpart;
        kb1 = min(kb0 + P.p[gi].kpart, kblocks);
        return part;
    };

    // K is consumed in chunks of KC blocks; each chunk accumulates in a fresh
    // TMEM buffer (two, alternating) and the epilogue warps add the chunk
    // results into FP32 registers, so no tensor-core accumulation chain is
    // longer than KC * 4 * (3 or 6) MMAs.
    constexpr int KC = 4;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&tail->full[s], 1);
            mbar_init(&tail->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tail->acc_full[b], 1);
            mbar_init(&tail->acc_empty[b], EW);  // one arrival per epilogue warp
        }
        mbar_init(&tail->mma_done, 1);
        tail->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tail->tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tail->tmem_base;
    volatile int *abort_flag = &tail->abort;
    const unsigned long long wlim = P.p[0].ep.wait_ns ? P.p[0].ep.wait_ns : kWaitNs;
    const int stall = P.p[0].ep.test_stall;  // tests: copies of the first stall - 1 blocks only

    if (warp == 0) {
        if (lane == 0) {
            int g = 0;  // k blocks issued by this CTA
            for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x) {
                int gi, lt, kb0, kb1;
                locate(tile, gi, lt, kb0, kb1);
                const TcProblem &pr = P.p[gi];
                const int n_ct = (pr.cols + BN - 1) / BN;
                const int row0 = (lt / n_ct) * BM, col0 = (lt % n_ct) * BN;
                for (int kb = kb0; kb < kb1; ++kb, ++g) {
                    int s = g % STAGES, r = g / STAGES;
                    if (!mbar_wait(&tail->empty[s], (r & 1) ^ 1, abort_flag, wlim)) {
                        *abort_flag = 1;
                        atomicOr(err, 1);
                        break;
                    }
                    if (stall && g >= stall - 1) continue;
                    unsigned char *st = smem + s * STAGE_BYTES;
                    mbar_expect_tx(&tail->full[s], STAGE_BYTES);
                    tma_load_2d(st, &pr.mA[0], &tail->full[s], kb * BK, row0);
                    tma_load_2d(st + A_BYTES, &pr.mA[1], &tail->full[s], kb * BK, row0);
                    if (NS == 3) tma_load_2d(st + 2 * A_BYTES, &pr.mA[2], &tail->full[s], kb * BK, row0);
                    tma_load_2d(st + NS * A_BYTES, &pr.mB[0], &tail->full[s], kb * BK, col0);
                    tma_load_2d(st + NS * A_BYTES + B_BYTES, &pr.mB[1], &tail->full[s], kb * BK, col0);
                    if (NS == 3) tma_load_2d(st + NS * A_BYTES + 2 * B_BYTES, &pr.mB[2], &tail->full[s], kb * BK, col0);
                }
            }
            // drain: wait until the consumer has released every slot we filled
            int last = g - 1;
            for (int kb = last - STAGES + 1 < 0 ? 0 : last - STAGES + 1; kb <= last && !*abort_flag; ++kb) {
                int s = kb % STAGES, r = kb / STAGES;
                if (!mbar_wait(&tail->empty[s], r & 1, abort_flag, wlim)) break;
            }
            wait_copies(tail->full, stall && g > stall - 1 ? stall - 1 : g, STAGES);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int g = 0, gc = 0;  // k blocks and K chunks consumed by this CTA
            int nchunks = 0;
            for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x, gc += nchunks) {
                int gi, lt, kb0, kb1;
                locate(tile, gi, lt, kb0, kb1);
                const int K = P.p[gi].K, cols = P.p[gi].cols;
                const int n_ct = (cols + BN - 1) / BN, kblocks = kb1 - kb0;
                nchunks = (kblocks + KC - 1) / KC;
                int ncol = cols - (lt % n_ct) * BN;
                if (ncol > BN) ncol = BN;
                const uint32_t idesc = idesc_bf16((ncol + 15) & ~15);
                for (int kb = 0; kb < kblocks; ++kb, ++g) {
                    const int q = gc + kb / KC, buf = q & 1, use = q >> 1;
                    const bool first = (kb % KC) == 0;
                    if (first && use >= 1 && !mbar_wait(&tail->acc_empty[buf], (use - 1) & 1, abort_flag, wlim)) {
                        *abort_flag = 1;
                        atomicOr(err, 8);
                        break;
                    }
                    int s = g % STAGES, r = g / STAGES;
                    if (!mbar_wait(&tail->full[s], r & 1, abort_flag, wlim)) {
                        *abort_flag = 1;
                        atomicOr(err, 2);
                        break;
                    }
                    tc_fence_after();
                    const uint32_t tacc = tmem + (uint32_t)(buf * BN);
                    uint32_t sa = smem_u32(smem + s * STAGE_BYTES);
                    uint32_t pa[3] = {sa, sa + A_BYTES, sa + 2 * A_BYTES};
                    uint32_t sb = sa + NS * A_BYTES;
                    uint32_t pb[3] = {sb, sb + B_BYTES, sb + 2 * B_BYTES};
                    int ksteps = (K - (kb0 + kb) * BK) / 16;
                    if (ksteps > BK / 16) ksteps = BK / 16;
                    for (int kk = 0; kk < ksteps; ++kk) {
                        uint32_t off = kk * 32;
                        uint32_t acc0 = (first && kk == 0) ? 0u : 1u;
                        // plane pairs (i, j) with i + j < NS, largest products first
                        umma(tacc, sdesc_sw128(pa[0] + off), sdesc_sw128(pb[0] + off), idesc, acc0);
                        umma(tacc, sdesc_sw128(pa[0] + off), sdesc_sw128(pb[1] + off), idesc, 1u);
                        umma(tacc, sdesc_sw128(pa[1] + off), sdesc_sw128(pb[0] + off), idesc, 1u);
                        if (NS == 3) {
                            umma(tacc, sdesc_sw128(pa[1] + off), sdesc_sw128(pb[1] + off), idesc, 1u);
                            umma(tacc, sdesc_sw128(pa[0] + off), sdesc_sw128(pb[2] + off), idesc, 1u);
                            umma(tacc, sdesc_sw128(pa[2] + off), sdesc_sw128(pb[0] + off), idesc, 1u);
                        }
                    }
                    umma_commit(&tail->empty[s]);
                    if ((kb % KC) == KC - 1 || kb == kblocks - 1) umma_commit(&tail->acc_full[buf]);
                }
            }
            wait_mmas(&tail->mma_done);
        }
    } else {
        // epilogue warps
        const int ew = warp - 2;
        const int quad = warp & 3;        // TMEM lane quadrant this warp may access
        const int half = ew >> 2;         // column group (a half for EW = 8)
        constexpr int HC = BN / NG;         // columns per group
        unsigned char *wst = staging + ew * 2 * kStagePlane;  // this warp's two W planes of 32 rows x 32 columns
        int gc = 0;                         // K chunks consumed by this CTA
        int nchunks = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, gc += nchunks) {
            int gi, lt, kb0, kb1;
            const int part = locate(tile, gi, lt, kb0, kb1);
            const TcEpilogue &ep = P.p[gi].ep;
            const int rows = P.p[gi].rows, cols = P.p[gi].cols;
            const int n_ct = (cols + BN - 1) / BN;
            nchunks = (kb1 - kb0 + KC - 1) / KC;
            const int rt = lt / n_ct, ct = lt % n_ct;
            const int row0 = rt * BM, col0 = ct * BN;
            int ncol = cols - col0;
            if (ncol > BN) ncol = BN;
            const int r = row0 + quad * 32 + lane;
            if (EPI == EPI_KERNEL || EPI == EPI_QPOW) {
                // stage the per-column constants while the MMAs run, after every
                // epilogue warp has finished with the previous tile's; a wait
                // that expired in one warp stops them all here
                ok = bar_and(4, kThreads - 64, ok);
                if (!ok) break;
                for (int c = threadIdx.x - 64; c < BN; c += kThreads - 64) {
                    // the column arrays are padded to 256; a 192-column tile
                    // can reach past them, where nothing is used
                    int cc = col0 + c;
                    col_s[c] = c < ncol ? ep.s_col[cc] : 0.f;
                    if (EPI == EPI_KERNEL) col_a[c] = c < ncol ? (float)ep.zeta * (ep.alpha_col[cc] * ep.d2) : 0.f;
                }
                named_barrier(3, kThreads - 64);
            }
            // promoted accumulation of the chunk results
            float acc[HC];
#pragma unroll
            for (int k = 0; k < HC; ++k) acc[k] = 0.f;
            for (int c = 0; c < nchunks; ++c) {
                const int q = gc + c, buf = q & 1, use = q >> 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&tail->acc_full[buf], use & 1, abort_flag, wlim));
                if (!ok) {
                    *abort_flag = 1;
                    if (lane == 0) atomicOr(err, 4);
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int ch = 0; ch < HC / 32; ++ch) {
                    int cbase = half * HC + ch * 32;
                    if (cbase < ncol) {
                        float v[32];
                        tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BN + cbase), v);
#pragma unroll
                        for (int k = 0; k < 32; ++k) acc[ch * 32 + k] += v[k];
                    }
                }
                tc_fence_before();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tail->acc_empty[buf]))
                                 : "memory");
            }
            if (!ok) {
                if (EPI == EPI_STORE) break;
                continue;  // to the barrier that stops every warp
            }
            if constexpr (EPI == EPI_KERNEL) {
                const float tr = r < rows ? ep.t_row[r] : 0.f;
                const bool store = ep.W_hi != nullptr && row0 + quad * 32 < rows;  // energies only: W is not needed
                float esum = 0.f, wsum = 0.f;
                // Z: zeta, or 0 for any
                auto kernel = [&](auto Z) {
#pragma unroll
                    for (int ch = 0; ch < HC / 32; ++ch) {
                        const int cbase = half * HC + ch * 32;  // column within tile
                        if (cbase >= ncol) continue;
                        uint32_t pl[NS][16];
#pragma unroll
                        for (int k = 0; k < 32; k += 4) {
                            const float4 s4 = *reinterpret_cast<const float4 *>(col_s + cbase + k);
                            const float4 a4 = *reinterpret_cast<const float4 *>(col_a + cbase + k);
                            const float sc[4] = {s4.x, s4.y, s4.z, s4.w}, ac[4] = {a4.x, a4.y, a4.z, a4.w};
                            float w[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const float q = acc[ch * 32 + k + u] + sc[u] + tr;
                                const float qz = Z.value == 4 ? (q * q) * q : powi_small(q, ep.zeta - 1);
                                w[u] = ac[u] * qz;
                                esum = fmaf(w[u], q, esum);
                                wsum += w[u];
                            }
#pragma unroll
                            for (int u = 0; u < 4; u += 2)
#pragma unroll
                                for (int p = 0; p < NS; ++p) {
                                    const __nv_bfloat162 h = __floats2bfloat162_rn(w[u], w[u + 1]);
                                    pl[p][(k + u) / 2] = *reinterpret_cast<const uint32_t *>(&h);
                                    const float2 hf = __bfloat1622float2(h);
                                    w[u] -= hf.x;
                                    w[u + 1] -= hf.y;
                                }
                        }
                        if (!store) continue;
#pragma unroll
                        for (int p0 = 0; p0 < NS; p0 += 2) {  // two planes at a time
                            if (lane == 0) bulk_wait_read();  // the staging's earlier stores have read it
                            __syncwarp();
#pragma unroll
                            for (int p = p0; p < NS && p < p0 + 2; ++p)
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    *reinterpret_cast<uint4 *>(wst + (p - p0) * kStagePlane + lane * 64 +
                                                               16 * (k ^ ((lane >> 1) & 3))) =
                                        make_uint4(pl[p][4 * k], pl[p][4 * k + 1], pl[p][4 * k + 2], pl[p][4 * k + 3]);
                            fence_async_shared();
                            __syncwarp();
                            if (lane == 0) {
#pragma unroll
                                for (int p = p0; p < NS && p < p0 + 2; ++p)
                                    tma_store_2d(&P.p[gi].mW[p], wst + (p - p0) * kStagePlane, col0 + cbase,
                                                 row0 + quad * 32);
                                bulk_commit();
                            }
                        }
                    }
                };
                if (ep.zeta == 4) kernel(std::integral_constant<int, 4>{});
                else kernel(std::integral_constant<int, 0>{});
                if (r < rows) {
                    const int slot = ct * NG + half;
                    ep.eps_part[(size_t)r * ep.n_part + slot] = esum / (float)ep.zeta;
                    ep.wsum_part[(size_t)r * ep.n_part + slot] = wsum;
                }
            } else if constexpr (EPI == EPI_QPOW) {
                const float tr = r < rows ? ep.t_row[r] : 0.f;
                const bool store = row0 + quad * 32 < rows;
                const float d2 = ep.d2, zd2 = (float)ep.zeta * d2;
                // Z: zeta, or 0 for any
                auto powers = [&](auto Z) {
#pragma unroll
                    for (int ch = 0; ch < HC / 32; ++ch) {
                        const int cbase = half * HC + ch * 32;  // column within tile
                        if (cbase >= ncol || !store) continue;
#pragma unroll
                        for (int p = 0; p < 2; ++p) {  // W', then k: 128-byte rows, 128-byte swizzle
                            if (lane == 0) bulk_wait_read();
                            __syncwarp();
#pragma unroll
                            for (int k = 0; k < 32; k += 4) {
                                const float4 s4 = *reinterpret_cast<const float4 *>(col_s + cbase + k);
                                const float sc[4] = {s4.x, s4.y, s4.z, s4.w};
                                float o[4];
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const float q = acc[ch * 32 + k + u] + sc[u] + tr;
                                    const float qz = Z.value == 4 ? (q * q) * q : powi_small(q, ep.zeta - 1);
                                    o[u] = p == 0 ? zd2 * qz : d2 * qz * q;
                                }
                                *reinterpret_cast<float4 *>(wst + lane * 128 + 16 * ((k >> 2) ^ (lane & 7))) =
                                    make_float4(o[0], o[1], o[2], o[3]);
                            }
                            fence_async_shared();
                            __syncwarp();
                            if (lane == 0) {
                                tma_store_2d(&P.p[gi].mW[p], wst, col0 + cbase, row0 + quad * 32);
                                bulk_commit();
                            }
                        }
                    }
                };
                if (ep.zeta == 4) powers(std::integral_constant<int, 4>{});
                else powers(std::integral_constant<int, 0>{});
            } else {
#pragma unroll
                for (int ch = 0; ch < HC / 32; ++ch) {
                    int cbase = half * HC + ch * 32;   // column within tile
                    if (cbase >= ncol || r >= rows) continue;
                    const float *v = acc + ch * 32;
                    int c0 = col0 + cbase;
                    int orow = ep.row_map ? ep.row_map[r] : r;
                    float *out = ep.C + ((size_t)part * rows + orow) * ep.ldc + c0;
                    if (cbase + 32 <= ncol && (ep.ldc & 3) == 0) {
#pragma unroll
                        for (int k = 0; k < 32; k += 4)
                            *reinterpret_cast<float4 *>(out + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
                    } else {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (cbase + k < ncol) out[k] = v[k];
                    }
                }
            }
        }
        if (EPI != EPI_STORE && lane == 0) bulk_wait_all();  // this warp's stores are done
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                     : "memory");
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

int sm_count()
{
    static int n[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 132;
    if (!n[dev]) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = 132;
        }
        n[dev] = v;
    }
    return n[dev];
}

// A row-major [rows][ld] array (cols of them valid) of BF16 or FP32, in boxes
// of box_rows x box_cols.
gap_status make_map(CUtensorMap *m, const void *ptr, int rows, int cols, int ld, int box_rows, int box_cols = BK,
                    CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B, bool fp32 = false)
{
    auto enc = encode_fn();
    if (!enc) {
        gap_set_error("cuTensorMapEncodeTiled is unavailable");
        return GAP_ECUDA;
    }
    const int item = fp32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(ptr) & 15) || ((long)ld * item) % 16) {
        gap_set_error("tensor map operand is not 16-byte aligned");
        return GAP_EINVAL;
    }
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * item};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(m, fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                     const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        gap_set_error("cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
        return GAP_ECUDA;
    }
    return GAP_OK;
}

template <int BN, int STAGES, int EPI, int NS, int G, int EW = kEpiWarps>
gap_status launch_g(const TcOperands *ops, const TcEpilogue *eps, int n, int *err, cudaStream_t st)
{
    TcProblems<G> P;
    memset(&P, 0, sizeof(P));
    long tiles = 0;
    for (int q = 0; q < n; ++q) {
        const TcOperands &op = ops[q];
        if (op.rows <= 0 || op.cols <= 0) continue;
        TcProblem &pr = P.p[P.n];
        const __nv_bfloat16 *A[3] = {op.A_hi, NS == 3 ? op.A_mid : op.A_lo, op.A_lo};
        const __nv_bfloat16 *B[3] = {op.B_hi, NS == 3 ? op.B_mid : op.B_lo, op.B_lo};
        for (int pl = 0; pl < 3; ++pl) {
            GAP_TRY(make_map(&pr.mA[pl], A[pl], op.rows, op.K, op.lda, BM));
            GAP_TRY(make_map(&pr.mB[pl], B[pl], op.cols, op.K, op.ldb, BN));
        }
        if (EPI == EPI_KERNEL && eps[q].W_hi) {
            const __nv_bfloat16 *W[3] = {eps[q].W_hi, NS == 3 ? eps[q].W_mid : eps[q].W_lo, eps[q].W_lo};
            for (int pl = 0; pl < NS; ++pl)
                GAP_TRY(make_map(&pr.mW[pl], W[pl], op.rows, eps[q].ldw, eps[q].ldw, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B));
        }
        if (EPI == EPI_QPOW) {
            float *out[2] = {eps[q].Wp, eps[q].kq};
            for (int p = 0; p < 2; ++p)
                GAP_TRY(make_map(&pr.mW[p], out[p], op.rows, eps[q].ldwp, eps[q].ldwp, 32, 32,
                                 CU_TENSOR_MAP_SWIZZLE_128B, true));
        }
        pr.rows = op.rows;
        pr.cols = op.cols;
        pr.K = op.K;
        pr.tile0 = (int)tiles;
        pr.ep = eps[q];
        const long per = (long)((op.cols + BN - 1) / BN) * ((op.rows + BM - 1) / BM);
        const int kblocks = (op.K + BK - 1) / BK, parts = EPI == EPI_STORE && op.ksplit > 1 ? op.ksplit : 1;
        const int chunks = (kblocks + 3) / 4;  // chunks of four K blocks (KC)
        pr.kpart = (chunks + parts - 1) / parts * 4;
        pr.tiles_part = (int)per;
        if ((long)(parts - 1) * pr.kpart >= kblocks || (long)parts * pr.kpart < kblocks) {
            gap_set_error("tensor-core GEMM: bad split of K");
            return GAP_EINVAL;
        }
        tiles += per * parts;
        ++P.n;
    }
    if (P.n == 0) return GAP_OK;
    if (tiles > 2147483647L) {
        gap_set_error("tensor-core GEMM: too many tiles");
        return GAP_EUNSUPPORTED;
    }
    P.n_tiles = (int)tiles;
    const size_t scratch = 2 * BN * sizeof(float), staging = EPI != EPI_STORE ? EW * 2 * kStagePlane : 0;
    // 896: the base is 128-byte aligned at least (the 256-column kernel-energy tile takes all 227 KB)
    const size_t shm = (size_t)STAGES * (NS * BM * BK * 2 + NS * BN * BK * 2) + staging +
                       ((sizeof(SharedTail) + 127) & ~size_t(127)) + scratch + 896;
    static_assert(STAGES * (NS * BM * BK * 2 + NS * BN * BK * 2) + (EPI != EPI_STORE ? EW * 2 * kStagePlane : 0) +
                          ((sizeof(SharedTail) + 127) & ~size_t(127)) + 2 * BN * sizeof(float) + 896 <=
                      227 * 1024,
                  "shared memory of a block");
    auto kern = k_tc_gemm<BN, STAGES, EPI, NS, G, EW>;
    GAP_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    dim3 grid((unsigned)(tiles < sm_count() ? tiles : sm_count()));
    gap_count_launch();
    kern<<<grid, 32 * (2 + EW), shm, st>>>(P, err);
    return gap_cuda_status(cudaGetLastError(), "k_tc_gemm");
}

template <int BN, int STAGES, int EPI, int NS>
gap_status launch(const TcOperands &op, const TcEpilogue &ep, int *err, cudaStream_t st)
{
    return launch_g<BN, STAGES, EPI, NS, 1>(&op, &ep, 1, err, st);
}

// Up to kMaxGroups problems in one launch (the default tile variant).
constexpr int kMaxGroups = 4;
template <int NS>
gap_status launch_grouped(const TcOperands *ops, const TcEpilogue *eps, int n, int epi, int *err, cudaStream_t st)
{
    constexpr int BN = NS == 3 ? 128 : 256;
    if (epi == EPI_KERNEL) return launch_g<BN, 2, EPI_KERNEL, NS, kMaxGroups>(ops, eps, n, err, st);
    if (epi == EPI_STORE) return launch_g<BN, 2, EPI_STORE, NS, kMaxGroups>(ops, eps, n, err, st);
    // 128 columns: a training batch of several species has few rows of each
    // (K_NM of 24 four-species boxes 804 -> 791 us, with the stores by TMA)
    if (epi == EPI_QPOW) return launch_g<128, 2, EPI_QPOW, NS, kMaxGroups>(ops, eps, n, err, st);
    gap_set_error("grouped tensor-core GEMM: bad epilogue");
    return GAP_EINVAL;
}

// Tile variants of the two-plane split: (column tile, TMA stages, epilogue
// warps).  The three-plane split has one (128, 2): its 96 KB stages leave
// room for two.  The last variant (192 columns, twelve epilogue warps in
// three column groups) exists for the kernel-energy and store epilogues.
struct TileVariant {
    int bn, stages, ew;
};
constexpr TileVariant kVariants2[] = {{256, 2, 8}, {128, 2, 8}, {128, 3, 8}, {192, 2, 12}};
constexpr int kNumVariants2 = 4;
constexpr int kVariantWide = 3;

bool variant_applies(int v, const TcOperands &op, int epi)
{
    return v < kVariantWide || (op.nsplit == 2 && (epi == EPI_KERNEL || epi == EPI_STORE));
}

template <int BN, int ST, int NS>
gap_status launch_bn(const TcOperands &op, const TcEpilogue &ep, int epi, int *err, cudaStream_t st)
{
    if (epi == EPI_KERNEL) return launch<BN, ST, EPI_KERNEL, NS>(op, ep, err, st);
    if (epi == EPI_QPOW) return launch<BN, ST, EPI_QPOW, NS>(op, ep, err, st);
    return launch<BN, ST, EPI_STORE, NS>(op, ep, err, st);
}

gap_status launch_variant(const TcOperands &op, const TcEpilogue &ep, int epi, int v, int *err, cudaStream_t st)
{
    if (op.nsplit == 3) return launch_bn<128, 2, 3>(op, ep, epi, err, st);
    if (v == kVariantWide) {
        if (!variant_applies(v, op, epi)) {
            gap_set_error("tile variant for the kernel-energy and store epilogues only");
            return GAP_EINVAL;
        }
        if (epi == EPI_KERNEL) return launch_g<192, 2, EPI_KERNEL, 2, 1, 12>(&op, &ep, 1, err, st);
        return launch_g<192, 2, EPI_STORE, 2, 1, 12>(&op, &ep, 1, err, st);
    }

    switch (v) {
    case 1: return launch_bn<128, 2, 2>(op, ep, epi, err, st);
    case 2: return launch_bn<128, 3, 2>(op, ep, epi, err, st);
    default: return launch_bn<256, 2, 2>(op, ep, epi, err, st);
    }
}

// Tile autotuner.  A shape class is (device, epilogue and whether it stores W,
// planes, K, columns, ceil(log2(rows))).  (Without the stores, an energies-only
// call, the kernel-energy epilogue is another load, and its tile decides how
// the energy partials are grouped.)  The first call of a class outside stream capture times
// every variant on that call's own operands and outputs (CUDA events on the
// call's stream: one warm-up launch, then the best of two) and keeps the
// fastest; every later call, and any call under capture, reuses the choice
// (the default variant while none is known).  All variants compute the same
// values; their outputs are rewritten by the call that follows.
struct TuneKey {
    int dev, epi, stores, nsplit, K, cols, rlog;
    bool operator<(const TuneKey &o) const
    {
        if (dev != o.dev) return dev < o.dev;
        if (epi != o.epi) return epi < o.epi;
        if (stores != o.stores) return stores < o.stores;
        if (nsplit != o.nsplit) return nsplit < o.nsplit;
        if (K != o.K) return K < o.K;
        if (cols != o.cols) return cols < o.cols;
        return rlog < o.rlog;
    }
};
struct TuneEntry {
    int variant;
    float ms[kNumVariants2];
};
std::mutex g_tune_mu;
std::map<TuneKey, TuneEntry> g_tune;
std::vector<std::pair<TuneKey, TuneEntry>> g_tune_log;  // in the order tuned

int rows_log2(int rows)
{
    int r = 0;
    while ((1 << r) < rows && r < 30) ++r;
    return r;
}

TuneKey tune_key(const TcOperands &op, const TcEpilogue &ep, int epi)
{
    int dev = 0;
    cudaGetDevice(&dev);
    return {dev, epi, epi != EPI_KERNEL || ep.W_hi ? 1 : 0, op.nsplit, op.K, op.cols, rows_log2(op.rows)};
}

// The column tile a variant uses for this call (the energy epilogue's
// partial sums are laid out per column tile).
TcEpilogue with_parts(const TcEpilogue &ep, int epi, const TcOperands &op, const TileVariant &tv)
{
    TcEpilogue e = ep;
    if (epi == EPI_KERNEL) e.n_part = tv.ew / 4 * ((op.cols + tv.bn - 1) / tv.bn);
    return e;
}

}  // namespace

int gap_tc_sm_count() { return sm_count(); }

int gap_tc_ksplit(long tiles, int K)
{
    const int chunks = (K + 4 * BK - 1) / (4 * BK);
    if (tiles <= 0 || chunks <= 1 || 2 * tiles > sm_count()) return 1;
    int parts = (int)(sm_count() / tiles);
    if (parts > chunks) parts = chunks;
    const int per = (chunks + parts - 1) / parts;  // chunks per part
    return (chunks + per - 1) / per;               // no empty part
}

gap_status gap_tc_make_map(CUtensorMap *m, const void *ptr, int rows, int cols, int ld, int box_rows)
{
    return make_map(m, ptr, rows, cols, ld, box_rows);
}

int gap_tc_max_parts(int cols)
{
    int m = 0;
    for (const TileVariant &tv : kVariants2) {
        const int p = tv.ew / 4 * ((cols + tv.bn - 1) / tv.bn);
        if (p > m) m = p;
    }
    return m;
}

namespace {
std::atomic<int> g_force_variant{-1};  // gap_tc_force_variant (test hook)

int forced_variant(const TcOperands &op, int epi)
{
    const int v = g_force_variant.load();
    return v >= 0 && v < kNumVariants2 && op.nsplit == 2 && variant_applies(v, op, epi) ? v : -1;
}
}  // namespace

void gap_tc_force_variant(int v) { g_force_variant.store(v < 0 ? -1 : v); }
bool gap_tc_variant_forced(int nsplit) { return nsplit == 2 && g_force_variant.load() >= 0; }

int gap_tc_plan(const TcOperands &op, const TcEpilogue &ep, int epi, int *err, cudaStream_t st, int *groups)
{
    if (groups) *groups = 2;
    if (const int fv = forced_variant(op, epi); fv >= 0) {
        if (groups) *groups = kVariants2[fv].ew / 4;
        return kVariants2[fv].bn;
    }
    if (op.nsplit == 3 || op.rows <= 0 || op.cols <= 0) return 128;
    if (ep.wait_ns) return kVariants2[0].bn;  // the timeout tests: nothing to time
    const TuneKey key = tune_key(op, ep, epi);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune.find(key);
        if (it != g_tune.end()) {
            if (groups) *groups = kVariants2[it->second.variant].ew / 4;
            return kVariants2[it->second.variant].bn;
        }
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return kVariants2[0].bn;
    }
    TuneEntry e{0, {}};
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        cudaGetLastError();
        return kVariants2[0].bn;
    }
    float best = 1e30f;
    for (int v = 0; v < kNumVariants2; ++v) {
        e.ms[v] = 1e30f;
        if (!variant_applies(v, op, epi)) {
            e.ms[v] = -1.f;  // not a candidate for this class
            continue;
        }
        const TcEpilogue ev = with_parts(ep, epi, op, kVariants2[v]);
        if (launch_variant(op, ev, epi, v, err, st) != GAP_OK) continue;
        for (int rep = 0; rep < 2; ++rep) {
            cudaEventRecord(e0, st);
            if (launch_variant(op, ev, epi, v, err, st) != GAP_OK) break;
            cudaEventRecord(e1, st);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ms < e.ms[v]) e.ms[v] = ms;
        }
        if (e.ms[v] < best) {
            best = e.ms[v];
            e.variant = v;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaGetLastError();
    std::lock_guard<std::mutex> lk(g_tune_mu);
    if (g_tune.emplace(key, e).second) g_tune_log.emplace_back(key, e);
    if (groups) *groups = kVariants2[e.variant].ew / 4;
    return kVariants2[e.variant].bn;
}

int gap_tc_tuned_count()
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    return (int)g_tune_log.size();
}

bool gap_tc_tuned_entry(int k, int *fields, float *ms)
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    if (k < 0 || k >= (int)g_tune_log.size()) return false;
    const TuneKey &key = g_tune_log[k].first;
    const TuneEntry &e = g_tune_log[k].second;
    const int f[8] = {key.epi, key.nsplit, key.K, key.cols, key.rlog, kVariants2[e.variant].bn,
                      kVariants2[e.variant].stages, key.dev};
    for (int i = 0; i < 8; ++i) fields[i] = f[i];
    for (int v = 0; v < kNumVariants2; ++v) ms[v] = e.ms[v];
    return true;
}

gap_status gap_tc_gemm(const TcOperands &op, const TcEpilogue &ep, int epi, int *err, cudaStream_t st)
{
    if (op.rows <= 0 || op.cols <= 0) return GAP_OK;
    if ((long)((op.rows + 127) / 128) * ((op.cols + 127) / 128 + 1) > 2147483647L) {
        gap_set_error("tensor-core GEMM: too many tiles");
        return GAP_EUNSUPPORTED;
    }
    if (op.K <= 0 || op.K % 16) {
        gap_set_error("tensor-core GEMM needs K to be a positive multiple of 16");
        return GAP_EINVAL;
    }
    if (op.nsplit == 3) {
        if (!op.A_mid || !op.B_mid) {
            gap_set_error("three-plane GEMM needs mid planes");
            return GAP_EINVAL;
        }
        return launch_variant(op, ep, epi, 0, err, st);
    }
    if (op.ksplit > 1) return launch_variant(op, ep, epi, 2, err, st);  // few 128 x 128 tiles
    if (const int fv = forced_variant(op, epi); fv >= 0)
        return launch_variant(op, with_parts(ep, epi, op, kVariants2[fv]), epi, fv, err, st);
    const int bn = gap_tc_plan(op, ep, epi, err, st);
    int v = 0;
    for (int k = 0; k < kNumVariants2; ++k)
        if (kVariants2[k].bn == bn) { v = k; break; }
    {
        // the planned variant (the plan returns its column tile; look up the
        // full entry for the stage count)
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune.find(tune_key(op, ep, epi));
        if (it != g_tune.end()) v = it->second.variant;
    }
    return launch_variant(op, with_parts(ep, epi, op, kVariants2[v]), epi, v, err, st);
}

int gap_tc_grouped_col_tile(int nsplit) { return nsplit == 3 ? 128 : 256; }

gap_status gap_tc_gemm_grouped(const TcOperands *ops, const TcEpilogue *eps, int n, int epi, int *err, cudaStream_t st)
{
    for (int q0 = 0; q0 < n; q0 += kMaxGroups) {
        const int m = n - q0 < kMaxGroups ? n - q0 : kMaxGroups;
        for (int q = q0; q < q0 + m; ++q) {
            if (ops[q].rows <= 0 || ops[q].cols <= 0) continue;
            if (ops[q].K <= 0 || ops[q].K % 16 || ops[q].nsplit != ops[q0].nsplit ||
                (ops[q].nsplit == 3 && (!ops[q].A_mid || !ops[q].B_mid))) {
                gap_set_error("grouped tensor-core GEMM: bad problem");
                return GAP_EINVAL;
            }
        }
        GAP_TRY(ops[q0].nsplit == 3 ? launch_grouped<3>(ops + q0, eps + q0, m, epi, err, st)
                                    : launch_grouped<2>(ops + q0, eps + q0, m, epi, err, st));
    }
    return GAP_OK;
}
