// K_NM force rows (text after Eq. 4) on the sm_103a tensor cores.
//
//   K[(j, a)][m] = sum_t W'[src t][m] (J_ta . (x_m - mu) + J_ta . mu),   t over the triples of target j
//
// One GEMM of the sparse points against the Jacobian rows, in split BF16
// (hi hi + hi lo + lo hi, FP32 accumulation in TMEM; six products with three
// planes), whose epilogue scales every column by its source's W' and sums the
// columns of a target.  The sparse points are the M side (a TMEM lane, so a
// thread, per sparse point) and the Jacobian rows the N side: a target's sum
// runs along a thread's own registers, W' rows are read 128 bytes per warp,
// and nothing is staged or exchanged between threads.  Rows come in triples
// that share one W', so a thread spends one W' load and six FP32
// instructions per three elements.
//
// The N side of a tile is NG groups of 48 rows (16 triples), each from its own
// stream: the triples of a range of targets.  Four epilogue warps serve a
// group (one per TMEM lane quadrant).  A CTA takes a work unit, one 128-point
// tile against NG ranges; ranges end between targets, so no group needs
// another's sums and every K entry is written once, complete.  A target's sum
// is FP32 over the triples of one tile (sixteen at most) and FP64 over its
// tiles, in shared memory (0.4% of K_NM of 200 silicon cells).  Units that
// share ranges differ in the point tile and run side by side, so a Jacobian row
// is read from HBM once and otherwise from L2.
//
// What bounds it is latency in the epilogue: one group over the whole tile
// (four warps, one per scheduler) takes 12 thousand cycles per tile where the
// MMAs take 4.6 thousand; with four groups each scheduler has four warps.
// W' rows and row data are loaded one and two tiles ahead.  K_NM of 200
// silicon cells (2.17 million rows, 2000 points, D = 252): 4.75 ms here, 7.4 ms
// with the rows on the M side, W' gathered per row and the target sums through
// shared memory; the MMAs and the TMEM reads alone take about 3.7 ms.
//
//   warp 0       TMA producer (one lane), K blocks of 64, STAGES-deep ring
//   warp 1       TMEM allocation, MMA issue (one lane)
//   warps 2 ..   epilogue
//
// K is consumed in chunks of 256 that each start a fresh accumulator (two,
// alternating); the epilogue adds the chunks in FP32 registers, so no
// tensor-core accumulation chain is longer.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstring>

#include "knm_gemm.h"
#include "tc_gemm.h"
#include "tc_prim.cuh"

namespace {

using namespace tcp;

constexpr int BM = 128, BK = 64, KC = 4;
constexpr int kGT = 16, kGC = 3 * kGT;  // triples and columns (rows of J) per group

struct KnmProblem {
    CUtensorMap mA[3];  // sparse points: hi, mid or lo, lo
    const float *Wp;
    int M, ld, col0;
    int n_mt, unit0;  // 128-point tiles, first unit
};
struct KnmParams {
    CUtensorMap mJ[3];
    KnmProblem p[kKnmMaxGPs];
    const float4 *meta;
    const int *dest, *bounds;  // bounds[problem][kMaxRanges + 1]
    double *K;
    long ldk;
    int n, n_units, kdim;
};
constexpr int kMaxRanges = 2048;

struct KnmTail {
    uint64_t full[4], empty[4], acc_full[2], acc_empty[2], mma_done;
    uint32_t tmem_base;
    int abort;
};

// 24 consecutive TMEM columns of this warp's lanes.
__device__ __forceinline__ void tmem_ld24(uint32_t taddr, float *v)
{
    uint32_t r[24];
#define R8(o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
    asm volatile(
        "{\n\t.reg .b32 t1;\n\tadd.u32 t1, %24, 16;\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%24];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16, %17, %18, %19, %20, %21, %22, %23}, [t1];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t}\n"
        : R8(0), R8(8), R8(16)
        : "r"(taddr)
        : "memory");
#undef R8
#pragma unroll
    for (int k = 0; k < 24; ++k) v[k] = __uint_as_float(r[k]);
}

// ONE: a single K chunk (K <= 256), read from TMEM in two halves of 24 columns
// so that four groups' 18 warps keep their 96 registers; else the chunks are
// summed in 48 registers, which three groups (14 warps, 128 registers) hold.
template <int NG, int NS, int STAGES, bool ONE>
__global__ void __launch_bounds__(64 + 128 * NG, 1) k_knm_gemm(const __grid_constant__ KnmParams P, int *err)
{
    static_assert(NS == 2 || NS == 3, "planes");
    constexpr int NB = NG * kGC;
    static_assert(NB % 16 == 0 && NB <= 256, "MMA columns");
    constexpr uint32_t TMEM_COLS = 2 * NB <= 256 ? 256 : 512;
    constexpr uint32_t A_BYTES = BM * BK * 2, G_BYTES = kGC * BK * 2, B_BYTES = NG * G_BYTES,
                       STAGE_BYTES = NS * (A_BYTES + B_BYTES);
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    KnmTail *tail = reinterpret_cast<KnmTail *>(smem + STAGES * STAGE_BYTES);
    // J . mu of the triples of two tiles, per epilogue warp; after them every
    // epilogue thread's sums of its current target over earlier tiles
    float4 *meta_s = reinterpret_cast<float4 *>(smem + STAGES * STAGE_BYTES + 256);
    constexpr int kEpi = 128 * NG;
    double *carry_s = reinterpret_cast<double *>(meta_s + 4 * NG * 2 * kGT);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&tail->full[s], 1);
            mbar_init(&tail->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tail->acc_full[b], 1);
            mbar_init(&tail->acc_empty[b], 4 * NG);  // one arrival per epilogue warp
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
    const int n_units = P.n_units, kblocks = (P.kdim + BK - 1) / BK, nchunks = ONE ? 1 : (kblocks + KC - 1) / KC;
    // unit -> (problem, point tile, bounds of its NG ranges); returns its tiles
    auto locate = [&](int u, int &g, int &mt, const int *&bd) {
        g = 0;
#pragma unroll
        for (int k = 1; k < kKnmMaxGPs; ++k)
            if (k < P.n && u >= P.p[k].unit0) g = k;
        const int lu = u - P.p[g].unit0, r = lu / P.p[g].n_mt;
        mt = lu - r * P.p[g].n_mt;
        bd = P.bounds + g * (kMaxRanges + 1) + r * NG;
        int longest = 0;
#pragma unroll
        for (int k = 0; k < NG; ++k) longest = max(longest, bd[k + 1] - bd[k]);
        return (longest + kGT - 1) / kGT;
    };

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;  // K blocks issued
            for (int u = blockIdx.x; u < n_units && !*abort_flag; u += gridDim.x) {
                int g, mt;
                const int *bd;
                const int tiles = locate(u, g, mt, bd);
                const KnmProblem &pr = P.p[g];
                int q[NG];
#pragma unroll
                for (int k = 0; k < NG; ++k) q[k] = 3 * bd[k];
                for (int t = 0; t < tiles && !*abort_flag; ++t) {
                    for (int kb = 0; kb < kblocks; ++kb, ++it) {
                        const int s = it % STAGES, r = it / STAGES;
                        if (!mbar_wait(&tail->empty[s], (r & 1) ^ 1, abort_flag)) {
                            *abort_flag = 1;
                            atomicOr(err, 1);
                            break;
                        }
                        unsigned char *sm = smem + s * STAGE_BYTES;
                        mbar_expect_tx(&tail->full[s], STAGE_BYTES);
#pragma unroll
                        for (int pl = 0; pl < NS; ++pl) {
                            tma_load_2d(sm + pl * A_BYTES, &pr.mA[pl], &tail->full[s], kb * BK, mt * BM);
#pragma unroll
                            for (int k = 0; k < NG; ++k)
                                tma_load_2d(sm + NS * A_BYTES + pl * B_BYTES + k * G_BYTES, &P.mJ[pl], &tail->full[s],
                                            kb * BK, q[k] + t * kGC);
                        }
                    }
                }
            }
            // drain: wait until the consumer has released every slot filled
            for (int k = it - STAGES < 0 ? 0 : it - STAGES; k < it && !*abort_flag; ++k)
                if (!mbar_wait(&tail->empty[k % STAGES], (k / STAGES) & 1, abort_flag)) break;
            wait_copies(tail->full, it, STAGES);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0, gc = 0;  // K blocks and K chunks consumed
            const uint32_t idesc = idesc_bf16(NB);
            for (int u = blockIdx.x; u < n_units && !*abort_flag; u += gridDim.x) {
                int g, mt;
                const int *bd;
                const int tiles = locate(u, g, mt, bd);
                for (int t = 0; t < tiles && !*abort_flag; ++t, gc += nchunks) {
                    for (int kb = 0; kb < kblocks; ++kb, ++it) {
                        const int ch = gc + kb / KC, buf = ch & 1, use = ch >> 1;
                        const bool first = (kb % KC) == 0;
                        if (first && use >= 1 && !mbar_wait(&tail->acc_empty[buf], (use - 1) & 1, abort_flag)) {
                            *abort_flag = 1;
                            atomicOr(err, 8);
                            break;
                        }
                        const int s = it % STAGES, r = it / STAGES;
                        if (!mbar_wait(&tail->full[s], r & 1, abort_flag)) {
                            *abort_flag = 1;
                            atomicOr(err, 2);
                            break;
                        }
                        tc_fence_after();
                        const uint32_t tacc = tmem + (uint32_t)(buf * NB);
                        const uint32_t sa = smem_u32(smem + s * STAGE_BYTES), sb = sa + NS * A_BYTES;
                        int ksteps = (P.kdim - kb * BK) / 16;
                        if (ksteps > BK / 16) ksteps = BK / 16;
                        for (int kk = 0; kk < ksteps; ++kk) {
                            const uint32_t off = kk * 32;
                            // plane pairs (i, j) with i + j < NS, largest products first
                            umma(tacc, sdesc_sw128(sa + off), sdesc_sw128(sb + off), idesc, (first && kk == 0) ? 0u : 1u);
                            umma(tacc, sdesc_sw128(sa + off), sdesc_sw128(sb + B_BYTES + off), idesc, 1u);
                            umma(tacc, sdesc_sw128(sa + A_BYTES + off), sdesc_sw128(sb + off), idesc, 1u);
                            if (NS == 3) {
                                umma(tacc, sdesc_sw128(sa + A_BYTES + off), sdesc_sw128(sb + B_BYTES + off), idesc, 1u);
                                umma(tacc, sdesc_sw128(sa + off), sdesc_sw128(sb + 2 * B_BYTES + off), idesc, 1u);
                                umma(tacc, sdesc_sw128(sa + 2 * A_BYTES + off), sdesc_sw128(sb + off), idesc, 1u);
                            }
                        }
                        umma_commit(&tail->empty[s]);
                        if ((kb % KC) == KC - 1 || kb == kblocks - 1) umma_commit(&tail->acc_full[buf]);
                    }
                }
            }
            wait_mmas(&tail->mma_done);
        }
    } else {
        const int quad = warp & 3, grp = (warp - 2) >> 2;  // TMEM lane quadrant, column group
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(grp * kGC);
        float4 *wmeta = meta_s + (warp - 2) * 2 * kGT;
        double *carry = carry_s + (threadIdx.x - 64);  // [three rows][kEpi]
        int gc = 0;  // K chunks consumed
        bool ok = true;
        for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
            int g, mt;
            const int *bd;
            const int tiles = locate(u, g, mt, bd);
            const KnmProblem &pr = P.p[g];
            const int m = mt * BM + quad * 32 + lane, ld = pr.ld, q1 = bd[grp + 1];
            int q = bd[grp];
            const bool mine = m < pr.M;
            const float *Wm = pr.Wp + m;  // m < M_pad: inside the padded row
            double *Kc = P.K + pr.col0 + m;
            // the current target's sums: FP32 over a tile's triples (sixteen at
            // most), FP64 over the tiles
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
            bool carried = false;  // earlier tiles of the target are in carry
            auto total = [&](int a, float s) { return carried ? carry[a * kEpi] + (double)s : (double)s; };
            float w[kGT];
            int dest = -1;
            // lane k < 16 holds triple k of a tile; past the range's end zeros
            float4 nm;
            int nd;
            auto load_meta = [&](int at) {
                const bool in = lane < kGT && at + lane < q1;
                nm = in ? P.meta[at + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
                nd = in ? P.dest[at + lane] : -1;
            };
            auto load_w = [&](float (&o)[kGT]) {
                const int src = __float_as_int(nm.w);
#pragma unroll
                for (int k = 0; k < kGT; ++k) o[k] = __ldg(Wm + (size_t)__shfl_sync(0xffffffffu, src, k) * ld);
            };
            __syncwarp();  // the previous unit's last tile is read
            load_meta(q);
            load_w(w);
            if (lane < kGT) wmeta[lane] = nm;
            dest = nd;
            load_meta(q + kGT);
            for (int t = 0; t < tiles; ++t, q += kGT, gc += nchunks) {
                // the next tile: its W' into flight, its data to shared memory; the one after: its data
                float wn[kGT];
                load_w(wn);
                __syncwarp();  // every lane has read the tile before, whose place this is
                if (lane < kGT) wmeta[((t + 1) & 1) * kGT + lane] = nm;
                const int next_dest = nd;
                load_meta(q + 2 * kGT);
                __syncwarp();
                const float4 *md = wmeta + (t & 1) * kGT;
                const unsigned ends = __ballot_sync(0xffffffffu, dest >= 0);
                // triples 8 h .. 8 h + 7 of the tile, their columns in v
                auto sum_half = [&](int h, const float *v) {
                    if (((ends >> (8 * h)) & 0xffu) == 0) {  // no target ends here
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float4 e = md[8 * h + k];
                            s0 = fmaf(w[8 * h + k], v[3 * k] + e.x, s0);
                            s1 = fmaf(w[8 * h + k], v[3 * k + 1] + e.y, s1);
                            s2 = fmaf(w[8 * h + k], v[3 * k + 2] + e.z, s2);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float4 e = md[8 * h + k];
                            s0 = fmaf(w[8 * h + k], v[3 * k] + e.x, s0);
                            s1 = fmaf(w[8 * h + k], v[3 * k + 1] + e.y, s1);
                            s2 = fmaf(w[8 * h + k], v[3 * k + 2] + e.z, s2);
                            if (ends & (1u << (8 * h + k))) {  // the target's last triple
                                const int d = __shfl_sync(0xffffffffu, dest, 8 * h + k);
                                if (mine) {
                                    double *o = Kc + (size_t)d * P.ldk;
                                    o[0] = total(0, s0);
                                    o[P.ldk] = total(1, s1);
                                    o[2 * P.ldk] = total(2, s2);
                                }
                                s0 = s1 = s2 = 0.f;
                                carried = false;
                            }
                        }
                    }
                };
                if constexpr (ONE) {
                    const int buf = gc & 1, use = gc >> 1;
                    ok = __all_sync(0xffffffffu, mbar_wait(&tail->acc_full[buf], use & 1, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                    float v[24];
                    tmem_ld24(tq + (uint32_t)(buf * NB), v);
                    sum_half(0, v);
                    tmem_ld24(tq + (uint32_t)(buf * NB + 24), v);
                    tc_fence_before();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tail->acc_empty[buf]))
                                     : "memory");
                    sum_half(1, v);
                } else {
                    float v[kGC];
#pragma unroll
                    for (int k = 0; k < kGC; ++k) v[k] = 0.f;
                    for (int c = 0; c < nchunks; ++c) {
                        const int ch = gc + c, buf = ch & 1, use = ch >> 1;
                        ok = __all_sync(0xffffffffu, mbar_wait(&tail->acc_full[buf], use & 1, abort_flag));
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float x[24];
                            tmem_ld24(tq + (uint32_t)(buf * NB + 24 * h), x);
#pragma unroll
                            for (int k = 0; k < 24; ++k) v[24 * h + k] += x[k];
                        }
                        tc_fence_before();
                        if (lane == 0)
                            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tail->acc_empty[buf]))
                                         : "memory");
                    }
                    if (!ok) break;
                    sum_half(0, v);
                    sum_half(1, v + 24);
                }
                if (!(ends >> (kGT - 1) & 1u)) {  // the target goes on in the next tile
                    carry[0] = total(0, s0);
                    carry[kEpi] = total(1, s1);
                    carry[2 * kEpi] = total(2, s2);
                    s0 = s1 = s2 = 0.f;
                    carried = true;
                }
#pragma unroll
                for (int k = 0; k < kGT; ++k) w[k] = wn[k];
                dest = next_dest;
            }
        }
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) atomicOr(err, 4);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                     : "memory");
    }
}

// Range r of GP g covers the triples of whole targets, about 1 / n_r of the
// GP's; bounds[g][r] is its first triple.
struct RangePlan {
    int gp[kKnmMaxGPs], n_r[kKnmMaxGPs];
};
__global__ void k_knm_ranges(int n, const int *__restrict__ first, RangePlan plan, int *__restrict__ bounds)
{
    const int g = blockIdx.x, n_r = plan.n_r[g];
    const int *f = first + (size_t)plan.gp[g] * n;
    const long base = f[0], total = f[n] - base;
    for (int r = threadIdx.x; r <= n_r; r += blockDim.x) {
        const long want = base + total * r / n_r;
        int lo = 0, hi = n;  // the first target that starts at or after `want`
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (f[mid] < want) lo = mid + 1;
            else hi = mid;
        }
        bounds[g * (kMaxRanges + 1) + r] = f[lo];
    }
}

// A warp per target atom j: the place of each neighbour's triple among those
// of j and the neighbour's GP (the own triple, of j's GP, comes first).
__global__ void __launch_bounds__(128)
k_knm_slots(int n, int n_gp, const int *__restrict__ offsets, const int *__restrict__ nbr_j,
            const int *__restrict__ gp_of_atom, int *__restrict__ slot, int *__restrict__ counts)
{
    const int j = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= n) return;
    int cnt = lane == gp_of_atom[j] ? 1 : 0;  // lane g: triples of GP g so far
    const int p1 = offsets[j + 1];
    for (int p0 = offsets[j]; p0 < p1; p0 += 32) {
        const int p = p0 + lane;
        const int g = p < p1 ? gp_of_atom[nbr_j[p]] : -2;
        const unsigned same = __match_any_sync(0xffffffffu, g);
        const int base = __shfl_sync(0xffffffffu, cnt, g >= 0 ? g : 0);
        if (g >= 0) slot[p] = base + __popc(same & ((1u << lane) - 1u));
        for (int k = 0; k < n_gp; ++k) {
            const int c = __popc(__ballot_sync(0xffffffffu, g == k));
            if (lane == k) cnt += c;
        }
    }
    if (lane < n_gp) counts[(size_t)lane * n + j] = cnt;
}

struct EnergyGPs {
    KnmGP gp[kKnmMaxGPs];
};
// Energy rows: block per (128 columns, configuration, GP).  The GP's rows are
// ascending atoms, so a configuration's are consecutive.
__global__ void __launch_bounds__(128)
k_knm_energy_tc(const int *__restrict__ cfg_off, EnergyGPs gps, double *__restrict__ K, long ldk)
{
    const KnmGP &gp = gps.gp[blockIdx.z];
    const int c = blockIdx.y, m = blockIdx.x * 128 + threadIdx.x;
    __shared__ int range[2];
    if (threadIdx.x < 2) {
        const int want = cfg_off[c + threadIdx.x];
        int lo = 0, hi = gp.R;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (gp.rows[mid] < want) lo = mid + 1;
            else hi = mid;
        }
        range[threadIdx.x] = lo;
    }
    __syncthreads();
    if (m >= gp.M) return;
    const float *kq = gp.kq + m;
    const int ld = gp.M_pad, i1 = range[1];
    int i = range[0];
    double s = 0.0;
    // eight loads in flight; FP32 terms summed in fours before the FP64 sum
    // (FP64 adds are the scarce unit)
    for (; i + 8 <= i1; i += 8) {
        float a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] = kq[(size_t)(i + u) * ld];
        s += (double)((a[0] + a[1]) + (a[2] + a[3]));
        s += (double)((a[4] + a[5]) + (a[6] + a[7]));
    }
    for (; i + 4 <= i1; i += 4)
        s += (double)((kq[(size_t)i * ld] + kq[(size_t)(i + 1) * ld]) + (kq[(size_t)(i + 2) * ld] + kq[(size_t)(i + 3) * ld]));
    for (; i < i1; ++i) s += (double)kq[(size_t)i * ld];
    K[(size_t)(c + 3 * (size_t)cfg_off[c]) * ldk + gp.col0 + m] = s;
}

template <int NG, int NS, int STAGES, bool ONE>
gap_status launch_knm(KnmParams &P, const KnmTriples &t, const KnmGP *gps, const RangePlan &plan, long n_triples,
                      int n, int *bounds, int *err, cudaStream_t st)
{
    const __nv_bfloat16 *J[3] = {t.hi, NS == 3 ? t.mid : t.lo, t.lo};
    for (int pl = 0; pl < NS; ++pl)
        GAP_TRY(gap_tc_make_map(&P.mJ[pl], J[pl], (int)(3 * n_triples), P.kdim, P.kdim, kGC));
    for (int k = 0; k < P.n; ++k) {
        const KnmGP &gp = gps[plan.gp[k]];
        const __nv_bfloat16 *B[3] = {gp.B_hi, NS == 3 ? gp.B_mid : gp.B_lo, gp.B_lo};
        for (int pl = 0; pl < NS; ++pl)
            GAP_TRY(gap_tc_make_map(&P.p[k].mA[pl], B[pl], gp.M, P.kdim, P.kdim, BM));
    }
    gap_count_launch();
    k_knm_ranges<<<P.n, 256, 0, st>>>(n, t.first, plan, bounds);
    GAP_TRY_CUDA(cudaGetLastError());
    const size_t shm = (size_t)STAGES * NS * (BM + NG * kGC) * BK * 2 + 256 +
                       4 * NG * 2 * kGT * sizeof(float4) + 3 * 128 * NG * sizeof(double) + 1024;
    auto kern = k_knm_gemm<NG, NS, STAGES, ONE>;
    GAP_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    const int sms = gap_tc_sm_count();
    gap_count_launch();
    kern<<<P.n_units < sms ? P.n_units : sms, 64 + 128 * NG, shm, st>>>(P, err);
    return gap_cuda_status(cudaGetLastError(), "k_knm_gemm");
}

}  // namespace

gap_status gap_knm_slots(int n, int n_gp, const int *offsets, const int *nbr_j, const int *gp_of_atom, int *slot,
                         int *counts, cudaStream_t st)
{
    if (n <= 0) return GAP_OK;
    gap_count_launch();
    k_knm_slots<<<(n + 3) / 4, 128, 0, st>>>(n, n_gp, offsets, nbr_j, gp_of_atom, slot, counts);
    return gap_cuda_status(cudaGetLastError(), "k_knm_slots");
}

size_t gap_knm_bounds_ints(int n_gp) { return (size_t)(n_gp > 0 ? n_gp : 1) * (kMaxRanges + 1); }

gap_status gap_knm_force_tc(const KnmTriples &t, long n_triples, int n, int K, int nsplit, const KnmGP *gps, int n_gp,
                            int *bounds, double *Kout, long ldk, int *err, cudaStream_t st)
{
    if (n_triples <= 0) return GAP_OK;
    if (K <= 0 || K % 16 || n_gp > kKnmMaxGPs || 3 * n_triples > 2147483647L) {
        gap_set_error("K_NM force rows: inner size, number of GPs or rows out of range");
        return GAP_EUNSUPPORTED;
    }
    KnmParams P;
    memset(&P, 0, sizeof(P));
    RangePlan plan{};
    P.meta = t.meta;
    P.dest = t.dest;
    P.bounds = bounds;
    P.K = Kout;
    P.ldk = ldk;
    P.kdim = K;
    const bool one = K <= KC * BK && nsplit == 2;
    const int NG = one ? 4 : 3;
    double weight[kKnmMaxGPs], total = 0.0;
    long atoms = 0;
    for (int s = 0; s < n_gp; ++s) atoms += gps[s].R;
    for (int s = 0; s < n_gp; ++s) {
        const KnmGP &gp = gps[s];
        if (gp.M <= 0 || gp.R <= 0) continue;
        KnmProblem &pr = P.p[P.n];
        plan.gp[P.n] = s;
        pr.Wp = gp.Wp;
        pr.M = gp.M;
        pr.ld = gp.M_pad;
        pr.col0 = gp.col0;
        pr.n_mt = (gp.M + BM - 1) / BM;
        weight[P.n] = (double)n_triples * gp.R / atoms;  // its triples, about
        total += weight[P.n] * pr.n_mt;
        ++P.n;
    }
    if (P.n == 0) return GAP_OK;
    // Ranges per GP: the GPs share w units per SM in proportion to their work;
    // w weighs the last wave's idle SMs against a range's partly filled last
    // tile.  (2000 points, 712 thousand triples: 16 point tiles, w = 2, 19 x NG
    // ranges.)
    const int sms = gap_tc_sm_count();
    double best = 1e300;
    int units_of[kKnmMaxGPs];
    for (int w = 1; w <= 8; ++w) {
        int nu[kKnmMaxGPs];  // range groups
        long units = 0;
        double longest = 0.0;
        for (int k = 0; k < P.n; ++k) {
            const double f = std::floor((double)sms * w * weight[k] / total + 1e-9);
            nu[k] = f < 1.0 ? 1 : f > kMaxRanges / NG ? kMaxRanges / NG : (int)f;
            units += (long)nu[k] * P.p[k].n_mt;
            const double tiles = std::ceil(weight[k] / (nu[k] * NG) / kGT) + 2.0;
            if (tiles > longest) longest = tiles;
        }
        const double cost = longest * std::ceil((double)units / sms);
        if (units <= 2147483647L && cost < best) {
            best = cost;
            for (int k = 0; k < P.n; ++k) units_of[k] = nu[k];
        }
    }
    for (int k = 0; k < P.n; ++k) {
        plan.n_r[k] = units_of[k] * NG;
        P.p[k].unit0 = P.n_units;
        P.n_units += units_of[k] * P.p[k].n_mt;
    }
    if (nsplit == 3) return launch_knm<3, 3, 2, false>(P, t, gps, plan, n_triples, n, bounds, err, st);
    if (one) return launch_knm<4, 2, 2, true>(P, t, gps, plan, n_triples, n, bounds, err, st);
    return launch_knm<3, 2, 3, false>(P, t, gps, plan, n_triples, n, bounds, err, st);
}

gap_status gap_knm_energy_tc(int n_configs, const int *cfg_off, const KnmGP *gps, int n_gp, double *Kout, long ldk,
                             cudaStream_t st)
{
    EnergyGPs e{};
    int k = 0, M = 0;
    for (int s = 0; s < n_gp; ++s)
        if (gps[s].M > 0) {
            e.gp[k++] = gps[s];
            if (gps[s].M > M) M = gps[s].M;
        }
    if (k == 0) return GAP_OK;
    // configurations on y, 65535 at a time
    for (int c0 = 0; c0 < n_configs; c0 += 65535) {
        const int nc = n_configs - c0 < 65535 ? n_configs - c0 : 65535;
        gap_count_launch();
        k_knm_energy_tc<<<dim3((M + 127) / 128, nc, k), 128, 0, st>>>(cfg_off + c0, e, Kout + (size_t)c0 * ldk, ldk);
        GAP_TRY_CUDA(cudaGetLastError());
    }
    return GAP_OK;
}
