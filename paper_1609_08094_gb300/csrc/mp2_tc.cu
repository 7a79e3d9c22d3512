// RI-MP2 correlation energy in mixed precision on the tcgen05 tensor cores, in
// two forms.  The first (up to v = MP2_GRAM_MAX_V, tcorr_mp2_create) forms g of
// a block of the problem as one Gram matrix and sums the energy in a second
// pass (mp2_gram_kernel, further down); the second, where the blocks do not fit
// its scratch (larger v, or little free memory), forms and sums g tile pair by
// tile pair:
// the paper's mixed-precision variant of the RI-MP2 kernel (Sec. 2.1, with
// the dgemm of the integral assembly done in reduced precision, Sec. 3),
// re-designed with the split-precision scheme of the (T) contractions.
//
//   E_MP2 = - sum_{ij} sum_{ab} g_aibj (2 g_aibj - g_ajbi) / (e_a + e_b - e_i - e_j),
//   g_aibj = sum_gamma C^gamma_ai C^gamma_bj          (Eqs. mp2_energy, eri_sym_decomp)
//
// over the occupied pairs i <= j (Eq. tasks_rimp2; i < j counts twice).  A
// work item is (pair, tile pair A <= B of 128 virtual indices).  Per 64-byte K
// chunk the producer loads C_i[A], C_j[B], C_j[A], C_i[B] (hi and lo planes
// of the K-major C^T, rows past v are TMA zero fill); the MMA thread forms
// G = C_i[A] C_j[B]^T (= g on A x B) and H = C_j[A] C_i[B]^T (= g on B x A,
// transposed) in two M = N = 128 TMEM accumulators with all four products
// lo*lo + hi*lo + lo*hi + hi*hi of each operand pair, each K block of MP_KB
// chunks in a fresh, double-buffered accumulator (smallest products first,
// hi*hi last, as in the (T) kernel: the tensor core's truncating accumulation
// then acts on the smallest partial sums).  Unlike the (T) contractions the
// lo*lo product is kept: for i = j the same-index elements g_aa are sums of
// squares, where the dropped lo^2 would bias g one-signedly by the mean
// square of the split's relative residual (~3e-6 with BF16; those elements
// carry most of E for small o); the kernel is bound by operand ingest, so
// the fourth product costs no time.  The epilogue warps fold every block into register totals
// with round-to-nearest FP32 adds, and at the end of the item form the energy
// terms of their (a, b): over A x B and B x A together -2 (g^2 + h^2) / eps and
// 2 g h / eps; a diagonal tile pair covers its block once, -2 g^2 / eps and
// g h / eps.  g never reaches memory.  Denominators and the item's terms are
// FP32, the running sums FP64; one FP64 partial pair per CTA, summed by the
// FP64 path's deterministic Kahan kernel.
//
// Kernel structure: one persistent CTA per SM, 10 warps.  Warp 0: TMA
// producer, a ring of 3 stages of 8 planes of 128 rows x 64 bytes (64 KB).
// Warp 1: TMEM allocation (512 columns: G and H of two K blocks) and the MMA
// issue.  Warps 2-9: two per TMEM lane quarter, 64 columns of G and of H
// each.  Warps 0 and 1 run whole, one elected lane issuing (tc_common.cuh): o=50,
// v=450, naux=1500 in BF16X3 took 4.37 ms with both in a branch on the lane
// number and 3.71 ms so.  Every mbarrier wait is bounded (wall clock): on expiry the kernel
// sets an error flag, stops all roles, waits (bounded) for its own copies in
// flight, frees TMEM and returns; the host reports TCORR_ETIMEOUT.
#include <mutex>

#include "tc_pair.cuh"

namespace tcorr {
namespace {

using namespace tcx;

constexpr int MP_BM = MP2_TC_TILE;          // virtual indices per tile: M = N = 128
constexpr int MP_ROW = 64;                  // K bytes per shared-memory row (SWIZZLE_64B span)
constexpr int MP_TILE = MP_BM * MP_ROW;     // 8 KB: one plane of one operand tile
constexpr int MP_STAGE = 8 * MP_TILE;       // C_i[A], C_j[B], C_j[A], C_i[B] x (hi, lo)
constexpr int MP_STAGES = 3;
constexpr int MP_SMEM = MP_STAGES * MP_STAGE + 1024;
constexpr int MP_THREADS = 320;
constexpr int MP_EPI = 256;                 // warps 2-9
constexpr int MP_KB = 2;                    // K chunks per TMEM accumulator block
constexpr int MP_HALF = MP_BM / 2;          // columns of G (and of H) per epilogue warp
static_assert(MP_KB < MP_STAGES, "a K block holds its stages until its last MMA is issued");
static_assert(4 * MP_BM <= 512, "G and H of two K blocks fill the 512 TMEM columns");
static_assert(MP_TILE % 1024 == 0, "planes keep the 64-byte swizzle pattern aligned");
// stage plane order
enum { P_AI_HI = 0, P_AI_LO, P_BJ_HI, P_BJ_LO, P_AJ_HI, P_AJ_LO, P_BI_HI, P_BI_LO };

template <int KIND>
__global__ void __launch_bounds__(MP_THREADS, 1) mp2_tc_kernel(const __grid_constant__ Mp2TcArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[MP_STAGES], bar_empty[MP_STAGES];
    __shared__ __align__(8) uint64_t bar_hfull[2], bar_hempty[2];
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_sh;
    __shared__ double red[MP_EPI / 32][2];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_dyn) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MP_STAGES; s++) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(smem_u32(&bar_hfull[b]), 1);
            mbar_init(smem_u32(&bar_hempty[b]), MP_EPI);
        }
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_holder)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;

    const int kch = MP_ROW / (KIND == 1 ? 4 : 2);  // K elements per chunk
    const int nch = a.nch;
    // D = F32, A/B = TF32 (2) or BF16 (1), K-major, M = N = 128
    constexpr uint32_t fmt = KIND == 1 ? 2u : 1u;
    constexpr uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(MP_BM >> 3) << 17) |
                               ((uint32_t)(MP_BM >> 4) << 24);
    double ej = 0.0, ek = 0.0;  // epilogue threads: weighted Coulomb and exchange sums

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        int last_phase[MP_STAGES];
        for (int s = 0; s < MP_STAGES; s++) last_phase[s] = -1;
        bool ok = true;
        for (int64_t it = blockIdx.x; it < a.items && ok; it += gridDim.x) {
            const int pr = (int)(it / a.ntp), tp = (int)(it % a.ntp);
            const int i = uni(a.pairs[2 * pr]), j = uni(a.pairs[2 * pr + 1]);
            const int A0 = uni(a.tiles[2 * tp]) * MP_BM, B0 = uni(a.tiles[2 * tp + 1]) * MP_BM;
            for (int ch = 0; ch < nch; ch++) {
                if (!wait_warp(smem_u32(&bar_empty[stage]), phase ^ 1u, &abort_sh)) {
                    if (lane == 0) fail(&abort_sh, a.err, DERR_TIMEOUT_EMPTY);
                    ok = false;
                    break;
                }
                const uint32_t full = smem_u32(&bar_full[stage]);
                last_phase[stage] = (int)phase;
                const uint32_t s = sbase + stage * MP_STAGE;
                const int k0 = ch * kch;
                if (elect_one()) {
                    mbar_expect_tx(full, (uint32_t)MP_STAGE);
                    tma_load_3d(s + P_AI_HI * MP_TILE, &a.map[0], full, k0, A0, i);
                    tma_load_3d(s + P_AI_LO * MP_TILE, &a.map[1], full, k0, A0, i);
                    tma_load_3d(s + P_BJ_HI * MP_TILE, &a.map[0], full, k0, B0, j);
                    tma_load_3d(s + P_BJ_LO * MP_TILE, &a.map[1], full, k0, B0, j);
                    tma_load_3d(s + P_AJ_HI * MP_TILE, &a.map[0], full, k0, A0, j);
                    tma_load_3d(s + P_AJ_LO * MP_TILE, &a.map[1], full, k0, A0, j);
                    tma_load_3d(s + P_BI_HI * MP_TILE, &a.map[0], full, k0, B0, i);
                    tma_load_3d(s + P_BI_LO * MP_TILE, &a.map[1], full, k0, B0, i);
                }
                __syncwarp();
                if (++stage == MP_STAGES) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok && lane == 0) {  // let this CTA's copies in flight land before exiting
            for (int s = 0; s < MP_STAGES; s++) {
                if (last_phase[s] < 0) continue;
                const uint64_t t0 = gtimer();
                while (!mbar_test(smem_u32(&bar_full[s]), (uint32_t)last_phase[s]) &&
                       gtimer() - t0 < WAIT_LIMIT_NS) {
                }
            }
        }
    } else if (warp == 1) {
        int stage = 0;
        uint32_t phase = 0;
        uint32_t hblk = 0;  // K blocks issued so far: buffer hblk & 1, phase (hblk >> 1) & 1
        bool ok = true;
        const uint32_t tm = uni(tmem);
        for (int64_t it = blockIdx.x; it < a.items && ok; it += gridDim.x) {
            for (int c0 = 0; c0 < nch && ok; c0 += MP_KB) {
                const int nb = min(MP_KB, nch - c0);
                const uint32_t buf = hblk & 1u;
                const uint32_t dG = tm + buf * (uint32_t)(2 * MP_BM), dH = dG + (uint32_t)MP_BM;
                const int st0 = stage;
                for (int cb = 0; cb < nb; cb++) {
                    int code = 0;
                    if (!wait_warp(smem_u32(&bar_full[stage]), phase, &abort_sh)) code = DERR_TIMEOUT_FULL;
                    else if (cb == 0 && !wait_warp(smem_u32(&bar_hempty[buf]), ((hblk >> 1) & 1u) ^ 1u, &abort_sh))
                        code = DERR_TIMEOUT_TMEM;
                    if (code) {
                        if (lane == 0) fail(&abort_sh, a.err, code);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // descriptor low words of the stage's planes (see mma_lo): one K
                    // step of 32 bytes is +2; the block's first products zero D
                    const uint32_t s = desc_lo(sbase + stage * MP_STAGE);
                    const uint32_t ai = s + P_AI_HI * (MP_TILE >> 4), bj = s + P_BJ_HI * (MP_TILE >> 4);
                    const uint32_t aj = s + P_AJ_HI * (MP_TILE >> 4), bi = s + P_BI_HI * (MP_TILE >> 4);
                    constexpr uint32_t LO = MP_TILE >> 4;  // hi plane -> lo plane
                    if (elect_one()) {
                        if (cb == 0) mma_lo<KIND, 1, false>(dG, ai + LO, bj + LO, idesc);
                        else mma_lo<KIND, 1, true>(dG, ai + LO, bj + LO, idesc);
                        mma_lo<KIND, 1, true>(dG, ai, bj + LO, idesc);
                        mma_lo<KIND, 1, true>(dG, ai + LO, bj, idesc);
                        if (cb == 0) mma_lo<KIND, 1, false>(dH, aj + LO, bi + LO, idesc);
                        else mma_lo<KIND, 1, true>(dH, aj + LO, bi + LO, idesc);
                        mma_lo<KIND, 1, true>(dH, aj, bi + LO, idesc);
                        mma_lo<KIND, 1, true>(dH, aj + LO, bi, idesc);
                        mma_lo<KIND, 1, true>(dG, ai + LO + 2, bj + LO + 2, idesc);
                        mma_lo<KIND, 1, true>(dG, ai + 2, bj + LO + 2, idesc);
                        mma_lo<KIND, 1, true>(dG, ai + LO + 2, bj + 2, idesc);
                        mma_lo<KIND, 1, true>(dH, aj + LO + 2, bi + LO + 2, idesc);
                        mma_lo<KIND, 1, true>(dH, aj + 2, bi + LO + 2, idesc);
                        mma_lo<KIND, 1, true>(dH, aj + LO + 2, bi + 2, idesc);
                    }
                    __syncwarp();
                    if (++stage == MP_STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                // the dominant hi*hi products of the block last; each stage is
                // released (commit: arrives once every MMA issued so far has
                // completed) right after its last product is issued
                if (elect_one()) {
                    int sj = st0;
                    for (int cb = 0; cb < nb; cb++) {
                        const uint32_t s = desc_lo(sbase + sj * MP_STAGE);
                        const uint32_t ai = s + P_AI_HI * (MP_TILE >> 4), bj = s + P_BJ_HI * (MP_TILE >> 4);
                        const uint32_t aj = s + P_AJ_HI * (MP_TILE >> 4), bi = s + P_BI_HI * (MP_TILE >> 4);
                        mma_lo<KIND, 1, true>(dG, ai, bj, idesc);
                        mma_lo<KIND, 1, true>(dH, aj, bi, idesc);
                        mma_lo<KIND, 1, true>(dG, ai + 2, bj + 2, idesc);
                        mma_lo<KIND, 1, true>(dH, aj + 2, bi + 2, idesc);
                        tc_commit(smem_u32(&bar_empty[sj]));
                        if (++sj == MP_STAGES) sj = 0;
                    }
                    tc_commit(smem_u32(&bar_hfull[buf]));
                }
                __syncwarp();
                hblk++;
            }
        }
    } else {
        const int wq = warp & 3;              // TMEM lane quarter of this warp
        const int half = (warp - 2) >> 2;     // column half of G and of H
        const int row = wq * 32 + lane;       // accumulator row = a in tile A
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        const int nhb = (nch + MP_KB - 1) / MP_KB;
        const int v = a.v;
        uint32_t hblk = 0;
        bool ok = true;
        for (int64_t it = blockIdx.x; it < a.items && ok; it += gridDim.x) {
            const int pr = (int)(it / a.ntp), tp = (int)(it % a.ntp);
            const int i = a.pairs[2 * pr], j = a.pairs[2 * pr + 1];
            const int A0 = a.tiles[2 * tp] * MP_BM, B0 = a.tiles[2 * tp + 1] * MP_BM;
            float tg[MP_HALF], th[MP_HALF];
#pragma unroll
            for (int c = 0; c < MP_HALF; c++) tg[c] = th[c] = 0.f;
            for (int hb = 0; hb < nhb; hb++) {
                const uint32_t buf = hblk & 1u;
                int good = 1;
                if (lane == 0) good = mbar_wait(smem_u32(&bar_hfull[buf]), (hblk >> 1) & 1u, &abort_sh) ? 1 : 0;
                good = __shfl_sync(0xffffffffu, good, 0);
                __syncwarp();
                if (!good) { ok = false; break; }
                tc_fence_after();
                const uint32_t tg0 = tmem + lane_off + buf * (uint32_t)(2 * MP_BM) + (uint32_t)(half * MP_HALF);
#pragma unroll
                for (int c16 = 0; c16 < MP_HALF / 16; c16++) {
                    uint32_t r[16], r2[16];
                    tc_ld16(tg0 + (uint32_t)(c16 * 16), r);
                    tc_ld16(tg0 + (uint32_t)(MP_BM + c16 * 16), r2);
                    tc_wait_ld();
#pragma unroll
                    for (int x = 0; x < 16; x++) tg[c16 * 16 + x] += __uint_as_float(r[x]);
#pragma unroll
                    for (int x = 0; x < 16; x++) th[c16 * 16 + x] += __uint_as_float(r2[x]);
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bar_hempty[buf]));
                hblk++;
            }
            if (!ok) {
                if (lane == 0) fail(&abort_sh, a.err, DERR_TIMEOUT_TMEM);
                break;
            }
            // energy terms of this thread's row a and 64 columns b
            const int ar = A0 + row;
            if (ar < v) {
                const float ea = (float)(a.eps_v[ar] - (a.eps_o[i] + a.eps_o[j]));
                const bool dg = (A0 == B0);
                const int b0 = B0 + half * MP_HALF;
                float sj = 0.f, sk = 0.f;
#pragma unroll
                for (int x = 0; x < MP_HALF; x++) {
                    if (b0 + x < v) {  // b grows with x
                        const float rd = 1.0f / (ea + a.eps_vf[b0 + x]);
                        const float g = tg[x], h = th[x];
                        if (!dg) {
                            sj = fmaf(-2.f * (g * g + h * h), rd, sj);
                            sk = fmaf(2.f * g * h, rd, sk);
                        } else {
                            sj = fmaf(-2.f * g * g, rd, sj);
                            sk = fmaf(g * h, rd, sk);
                        }
                    }
                }
                const double w = (i == j) ? 1.0 : 2.0;  // the pair (j, i) has the same energy
                ej += w * (double)sj;
                ek += w * (double)sk;
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            ej += __shfl_xor_sync(0xffffffffu, ej, off);
            ek += __shfl_xor_sync(0xffffffffu, ek, off);
        }
        if (lane == 0) { red[warp - 2][0] = ej; red[warp - 2][1] = ek; }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {  // fixed order: the CTA's partial is deterministic
        double sj = 0.0, sk = 0.0;
        for (int w = 0; w < MP_EPI / 32; w++) { sj += red[w][0]; sk += red[w][1]; }
        a.partials[2 * blockIdx.x] = sj;
        a.partials[2 * blockIdx.x + 1] = sk;
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                     : "memory");
    }
}


// ---- Gram form ----------------------------------------------------------------
//
// With the rows (i, a) of C^T flattened, every g_aibj is an element of one Gram
// matrix X X^T, of which the part j >= i is needed: full 256 x 256 tiles of it
// have no padding but at the matrix edge, no tile is computed twice, and an SM
// takes in 64 KB per K block (128 rows of X twice, hi and lo) for 16 MMAs of M =
// 256, N = 256.  The tile-pair kernel above pads v to tiles of 128 (450 -> 512),
// computes G and H = G^T of diagonal tiles, and takes in 128 KB per K block for
// the same tensor work: at o=50, v=450, naux=1500 it forms 4.2e8 products x naux
// against 2.6e8.  There, in BF16X3, the tile-pair kernel took 3.71 ms; the Gram
// tiles take 1.62 ms (1.88 PFLOP/s of the four products) and the energy pass 0.54.
// g goes to a scratch of at most 1 GiB (one wave per so much of
// the problem) in FP32, as the register totals hold it, and the energy kernel
// reads the two tiles (i, A) x (j, B) and (i, B) x (j, A) that hold g_ab and g_ba.  The accumulation (four products, fresh accumulator per K block,
// register totals) is that of the tile-pair kernel; the roles and hand-offs are
// those of the SM-pair contraction (gemm_tc.cu).
constexpr int GR_STAGE = 4 * PAIR_A;      // A hi, lo, B hi, lo: 128 rows x 128 bytes each
constexpr int GR_STAGES = 3;
constexpr int GR_SMEM = GR_STAGES * GR_STAGE + 1024;
constexpr int GR_THREADS = 64 + PAIR_EPI;

// the four products of one K block (two chunks of two K steps): a, b: descriptor
// low words of the stage's A_hi and B_hi planes (lo: + LO), one K step is + 2
template <int KIND>
__device__ __forceinline__ void gram_block(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc) {
    constexpr uint32_t LO = PAIR_A >> 4;
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        if (k == 0) mma_lo<KIND, 2, false, DESC_HI128>(d, a + LO, b + LO, idesc);
        else mma_lo<KIND, 2, true, DESC_HI128>(d, a + LO + k, b + LO + k, idesc);
        mma_lo<KIND, 2, true, DESC_HI128>(d, a + k, b + LO + k, idesc);
        mma_lo<KIND, 2, true, DESC_HI128>(d, a + LO + k, b + k, idesc);
    }
#pragma unroll
    for (int k = 0; k < 8; k += 2) mma_lo<KIND, 2, true, DESC_HI128>(d, a + k, b + k, idesc);
}

template <int KIND>
__global__ void __launch_bounds__(GR_THREADS, 1) mp2_gram_kernel(const __grid_constant__ Mp2GramArgs p,
                                                                 const __grid_constant__ Mp2Wave w) {
    extern __shared__ __align__(1024) uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[GR_STAGES], bar_empty[GR_STAGES];
    __shared__ __align__(8) uint64_t bar_hfull[2], bar_hempty[2];
    __shared__ __align__(8) uint64_t bar_fin;
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank(), cid = cluster_id(), ncl = cluster_count();
    const bool leader = rank == 0;
    const uint32_t sbase = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t peer_abort = peer_addr(smem_u32((const void *)&abort_sh), rank ^ 1u);

    if (threadIdx.x == 0) {
        for (int s = 0; s < GR_STAGES; s++) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(smem_u32(&bar_hfull[b]), 1);
            mbar_init(smem_u32(&bar_hempty[b]), PAIR_HEMPTY_ARRIVALS);
        }
        mbar_init(smem_u32(&bar_fin), 1);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_holder)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist before any remote signal
    tc_fence_after();
    const uint32_t tmem = tmem_holder;
    // D = F32, A/B = TF32 (2) or BF16 (1), K-major, M = 256 over the pair, N = 256
    constexpr uint32_t fmt = KIND == 1 ? 2u : 1u;
    constexpr uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(MP2_GRAM_TILE >> 3) << 17) |
                               ((uint32_t)(MP2_GRAM_TILE >> 4) << 24);
    const int nblk = p.nblk;

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        int last_phase[GR_STAGES];
        for (int s = 0; s < GR_STAGES; s++) last_phase[s] = -1;
        bool ok = true;
        for (int it = (int)cid; it < w.ntile && ok; it += (int)ncl) {
            const int2 t = p.tiles[w.tile0 + it];
            const int ra = uni((int)(w.row0 + (int64_t)t.x * MP2_GRAM_TILE) + (int)rank * PAIR_BM);
            const int rb = uni((int)(w.col0 + (int64_t)t.y * MP2_GRAM_TILE) + (int)rank * PAIR_BM);
            for (int kb = 0; kb < nblk; kb++) {
                if (!wait_warp(smem_u32(&bar_empty[stage]), phase ^ 1u, &abort_sh)) {
                    if (lane == 0) fail_pair(&abort_sh, peer_abort, p.err, DERR_TIMEOUT_EMPTY);
                    ok = false;
                    break;
                }
                const uint32_t full = smem_u32(&bar_full[stage]);
                const uint32_t full_l = peer_addr(full, 0);
                last_phase[stage] = (int)phase;
                const uint32_t s = sbase + stage * GR_STAGE;
                const int k0 = kb * (PAIR_ROW / (KIND == 1 ? 4 : 2));
                if (elect_one()) {
                    if (leader) mbar_expect_tx(full, 2u * (uint32_t)GR_STAGE);  // both CTAs' bytes
                    tma_load_2d_pair(s, &p.map[0], full_l, k0, ra);
                    tma_load_2d_pair(s + PAIR_A, &p.map[1], full_l, k0, ra);
                    tma_load_2d_pair(s + 2 * PAIR_A, &p.map[0], full_l, k0, rb);
                    tma_load_2d_pair(s + 3 * PAIR_A, &p.map[1], full_l, k0, rb);
                }
                __syncwarp();
                if (++stage == GR_STAGES) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok && lane == 0) {
            // let the copies in flight land: the leader sees both CTAs' bytes on
            // its own full barriers; the peer gives its own copies a fixed time
            if (leader) {
                for (int s = 0; s < GR_STAGES; s++) {
                    if (last_phase[s] < 0) continue;
                    const uint64_t t0 = gtimer();
                    while (!mbar_test(smem_u32(&bar_full[s]), (uint32_t)last_phase[s]) &&
                           gtimer() - t0 < WAIT_LIMIT_NS) {
                    }
                }
            }
            spin_ns(1000000ull);
        }
    } else if (warp == 1) {
        if (leader) {
            int stage = 0;
            uint32_t phase = 0, hblk = 0;
            bool ok = true;
            const uint32_t tm = uni(tmem);
            for (int it = (int)cid; it < w.ntile && ok; it += (int)ncl) {
                for (int kb = 0; kb < nblk; kb++) {
                    const uint32_t buf = hblk & 1u;
                    int code = 0;
                    if (!wait_warp(smem_u32(&bar_full[stage]), phase, &abort_sh)) code = DERR_TIMEOUT_FULL;
                    else if (!wait_warp(smem_u32(&bar_hempty[buf]), ((hblk >> 1) & 1u) ^ 1u, &abort_sh))
                        code = DERR_TIMEOUT_TMEM;
                    if (code) {
                        if (lane == 0) fail_pair(&abort_sh, peer_abort, p.err, code);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = desc_lo(sbase + stage * GR_STAGE), b = a + 2 * (PAIR_A >> 4);
                    if (elect_one()) {
                        gram_block<KIND>(tm + buf * (uint32_t)MP2_GRAM_TILE, a, b, idesc);
                        tc_commit_pair(smem_u32(&bar_empty[stage]), (uint16_t)3);
                        tc_commit_pair(smem_u32(&bar_hfull[buf]), (uint16_t)3);
                    }
                    __syncwarp();
                    if (++stage == GR_STAGES) { stage = 0; phase ^= 1u; }
                    hblk++;
                }
            }
            // every MMA issued by this warp's elected lane has completed before the pair tears down
            if (elect_one()) {
                tc_commit_pair(smem_u32(&bar_fin), (uint16_t)1);
                const uint64_t t0 = gtimer();
                while (!mbar_test(smem_u32(&bar_fin), 0u) && gtimer() - t0 < WAIT_LIMIT_NS) {
                }
            }
            __syncwarp();
        }
    } else {
        const int wq = warp & 3;              // TMEM lane quarter of this warp
        const int half = (warp - 2) >> 2;     // column half of the accumulator
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        uint32_t hblk = 0;
        bool ok = true;
        for (int it = (int)cid; it < w.ntile && ok; it += (int)ncl) {
            float total[128];
#pragma unroll
            for (int j = 0; j < 128; j++) total[j] = 0.f;
            for (int hb = 0; hb < nblk; hb++) {
                const uint32_t buf = hblk & 1u;
                if (!wait_warp(smem_u32(&bar_hfull[buf]), (hblk >> 1) & 1u, &abort_sh)) {
                    if (lane == 0) fail_pair(&abort_sh, peer_abort, p.err, DERR_TIMEOUT_TMEM);
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int c4 = 0; c4 < 4; c4++) {
                    uint32_t r[16], r2[16];
                    const uint32_t ta = tmem + lane_off + buf * (uint32_t)MP2_GRAM_TILE + (uint32_t)(half * 128 + c4 * 32);
                    tc_ld16(ta, r);
                    tc_ld16(ta + 16, r2);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; j++) total[c4 * 32 + j] += __uint_as_float(r[j]);
#pragma unroll
                    for (int j = 0; j < 16; j++) total[c4 * 32 + 16 + j] += __uint_as_float(r2[j]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(peer_addr(smem_u32(&bar_hempty[buf]), 0));
                hblk++;
            }
            if (!ok) break;
            const int2 t = p.tiles[w.tile0 + it];
            const int64_t r = (int64_t)t.x * MP2_GRAM_TILE + rank * PAIR_BM + wq * 32 + lane;
            const int64_t c0 = (int64_t)t.y * MP2_GRAM_TILE + half * 128;
            if (r < w.nrows) {
                float *out = p.g + r * w.ld + c0;  // 32-byte aligned: ld and c0 are multiples of 8
#pragma unroll
                for (int k = 0; k < 16; k++)  // values past ncols are products with zero rows or the next columns
                    if (c0 + 8 * k < w.ncols) st_v8(out + 8 * k, total + 8 * k);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // the peer no longer signals this CTA's barriers or reads its operands
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                     : "memory");
    }
}

// Energy of a wave's pairs from its stored g.  A work item is (pair i <= j, tile
// pair A <= B of 128 virtual indices, half of B): thread a of 128 sums the terms
// of its row a over 64 columns b in FP32, in the order of the tile-pair kernel,
// then in FP64.  g_ab comes through shared memory (read by rows, used by
// columns), g_ba = g of (i, B) x (j, A) is read by the threads side by side.  One
// FP64 partial pair per CTA.  Bound by reading g once.
constexpr int GE_T = MP2_TC_TILE;   // rows: threads
constexpr int GE_H = GE_T / 2;      // columns
constexpr int GE_CTAS = 5;          // per SM (the registers of 64 loads in flight)
__global__ void __launch_bounds__(GE_T, GE_CTAS) mp2_energy_kernel(const __grid_constant__ Mp2GramArgs p,
                                                                   const __grid_constant__ Mp2Wave w) {
    __shared__ float gs[GE_T][GE_H + 1];
    __shared__ float ev[GE_H];
    __shared__ double red[GE_T / 32][2];
    const int v = p.v, nt = (v + GE_T - 1) / GE_T, nit = nt * (nt + 1);  // tile pairs x halves
    const int tid = threadIdx.x;
    double ej = 0.0, ek = 0.0;
    const int64_t items = (int64_t)w.npair * nit;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t pr = w.pair0 + it / nit;
        int tp = (int)(it % nit), A = 0;
        const int half = tp & 1;
        tp >>= 1;
        while (tp >= nt - A) { tp -= nt - A; A++; }
        const int a0 = A * GE_T, b0 = (A + tp) * GE_T + half * GE_H;
        const bool dg = tp == 0;
        const int nb = min(GE_H, v - b0), na = min(GE_T, v - a0);
        if (nb <= 0) continue;
        const int i = p.pairs[2 * pr], j = p.pairs[2 * pr + 1];
        const float *G = p.g + ((int64_t)i * v - w.row0 + a0) * w.ld + ((int64_t)j * v - w.col0 + b0);
        const float *H = p.g + ((int64_t)i * v - w.row0 + b0) * w.ld + ((int64_t)j * v - w.col0 + a0) + tid;
        __syncthreads();  // the previous item's reads of gs
        // every load of the item in flight at once: G into shared memory, H in registers
        {
            const int c = tid & (GE_H - 1), r0 = tid / GE_H;
            if (c < nb) {
                const uint32_t dst = smem_u32(&gs[r0][c]);
                const float *src = G + (int64_t)r0 * w.ld + c;
#pragma unroll
                for (int k = 0; k < GE_T * GE_H / GE_T; k++)
                    if (r0 + (GE_T / GE_H) * k < na)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                         dst + (uint32_t)(k * (GE_T / GE_H) * (GE_H + 1) * 4)),
                                     "l"(src + (int64_t)k * (GE_T / GE_H) * w.ld)
                                     : "memory");
            }
        }
        float h[GE_H];
#pragma unroll
        for (int x = 0; x < GE_H; x++) h[x] = (tid < na && x < nb) ? H[(int64_t)x * w.ld] : 0.f;
        if (tid < GE_H) ev[tid] = tid < nb ? p.eps_vf[b0 + tid] : 1.f;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (tid < na) {
            const float ea = (float)(p.eps_v[a0 + tid] - (p.eps_o[i] + p.eps_o[j]));
            float sj = 0.f, sk = 0.f;
#pragma unroll
            for (int x = 0; x < GE_H; x++) {
                if (x < nb) {
                    const float rd = __frcp_rn(ea + ev[x]);  // = 1 / (ea + ev[x])
                    const float g = gs[tid][x];
                    if (!dg) {
                        sj = fmaf(-2.f * (g * g + h[x] * h[x]), rd, sj);
                        sk = fmaf(2.f * g * h[x], rd, sk);
                    } else {
                        sj = fmaf(-2.f * g * g, rd, sj);
                        sk = fmaf(g * h[x], rd, sk);
                    }
                }
            }
            const double wt = (i == j) ? 1.0 : 2.0;  // the pair (j, i) has the same energy
            ej += wt * (double)sj;
            ek += wt * (double)sk;
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        ej += __shfl_xor_sync(0xffffffffu, ej, off);
        ek += __shfl_xor_sync(0xffffffffu, ek, off);
    }
    if ((tid & 31) == 0) { red[tid >> 5][0] = ej; red[tid >> 5][1] = ek; }
    __syncthreads();
    if (tid == 0) {  // fixed order: the CTA's partial is deterministic
        double sj = 0.0, sk = 0.0;
        for (int n = 0; n < GE_T / 32; n++) { sj += red[n][0]; sk += red[n][1]; }
        p.partials[2 * (w.part0 + (int)blockIdx.x)] = sj;
        p.partials[2 * (w.part0 + (int)blockIdx.x) + 1] = sk;
    }
}

}  // namespace

using tcx::encode;

cudaError_t mp2_tc_fill(Mp2TcArgs &a, int prec, void *hi, void *lo, int o, int v, int kp, std::string &err) {
    const bool tf = prec == TCORR_TF32X3;
    const uint64_t eb = tf ? 4 : 2;
    const int kch = MP_ROW / (int)eb;
    if (kp % kch != 0) {
        err = "RI-MP2 tensor-core path: K extent not a multiple of the chunk";
        return cudaErrorInvalidValue;
    }
    const CUtensorMapDataType dt = tf ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    // Ct[i][a][gamma]: (gamma, a, i), rows past v read as zeros
    uint64_t dims[3] = {(uint64_t)kp, (uint64_t)v, (uint64_t)o};
    uint64_t st[2] = {(uint64_t)kp * eb, (uint64_t)v * kp * eb};
    uint32_t box[3] = {(uint32_t)kch, (uint32_t)MP_BM, 1};
    if (!encode(&a.map[0], dt, 3, hi, dims, st, box, err, "C hi")) return cudaErrorInvalidValue;
    if (!encode(&a.map[1], dt, 3, lo, dims, st, box, err, "C lo")) return cudaErrorInvalidValue;
    a.nch = kp / kch;
    return cudaSuccess;
}

cudaError_t launch_mp2_tc(int prec, int sm_count, const Mp2TcArgs &a, cudaStream_t st) {
    static std::mutex mu;
    static bool done[2] = {false, false};
    const int t = prec == TCORR_TF32X3 ? 0 : 1;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!done[t]) {
            const cudaError_t e =
                t == 0 ? cudaFuncSetAttribute(mp2_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MP_SMEM)
                       : cudaFuncSetAttribute(mp2_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MP_SMEM);
            if (e != cudaSuccess) return e;
            done[t] = true;
        }
    }
    const int grid = (int)std::min<int64_t>(sm_count, a.items);
    if (grid <= 0) return cudaSuccess;
    if (t == 0) mp2_tc_kernel<1><<<grid, MP_THREADS, MP_SMEM, st>>>(a);
    else mp2_tc_kernel<2><<<grid, MP_THREADS, MP_SMEM, st>>>(a);
    return cudaGetLastError();
}

cudaError_t mp2_gram_fill(Mp2GramArgs &a, int prec, void *hi, void *lo, int o, int v, int kp, std::string &err) {
    const bool tf = prec == TCORR_TF32X3;
    const uint64_t eb = tf ? 4 : 2;
    const int kblk = PAIR_ROW / (int)eb;
    const CUtensorMapDataType dt = tf ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    uint64_t dims[2] = {(uint64_t)kp, (uint64_t)o * v};
    uint64_t st[1] = {(uint64_t)kp * eb};
    uint32_t box[2] = {(uint32_t)kblk, (uint32_t)PAIR_BM};
    for (int n = 0; n < 2; n++)
        if (!encode(&a.map[n], dt, 2, n == 0 ? hi : lo, dims, st, box, err, n == 0 ? "C rows hi" : "C rows lo",
                    CU_TENSOR_MAP_SWIZZLE_128B))
            return cudaErrorInvalidValue;
    a.nblk = (kp + kblk - 1) / kblk;
    return cudaSuccess;
}

cudaError_t launch_mp2_gram(int prec, int sm_count, const Mp2GramArgs &a, const Mp2Wave &w, cudaStream_t st) {
    static std::mutex mu;
    static bool done = false;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!done) {
            cudaError_t e =
                cudaFuncSetAttribute(mp2_gram_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, GR_SMEM);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(mp2_gram_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, GR_SMEM);
            if (e != cudaSuccess) return e;
            done = true;
        }
    }
    static PairLaunch pl[2];
    return prec == TCORR_TF32X3 ? pl[0].launch(mp2_gram_kernel<1>, GR_THREADS, GR_SMEM, sm_count, w.ntile, st, a, w)
                                : pl[1].launch(mp2_gram_kernel<2>, GR_THREADS, GR_SMEM, sm_count, w.ntile, st, a, w);
}

int mp2_energy_ctas(int sm_count, int v, int npair) {
    const int64_t nt = (v + GE_T - 1) / GE_T;
    return (int)std::min<int64_t>((int64_t)sm_count * GE_CTAS, (int64_t)npair * nt * (nt + 1));
}

cudaError_t launch_mp2_energy(int sm_count, const Mp2GramArgs &a, const Mp2Wave &w, cudaStream_t st) {
    const int grid = mp2_energy_ctas(sm_count, a.v, w.npair);
    if (grid <= 0) return cudaSuccess;
    mp2_energy_kernel<<<grid, GE_T, 0, st>>>(a, w);
    return cudaGetLastError();
}

}  // namespace tcorr
