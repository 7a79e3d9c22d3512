// FP64-accurate W contractions on the BF16 tensor cores (Ozaki scheme,
// Ozaki et al. 2012; Mukunoki et al. 2020 on tensor cores): the same grouped
// GEMMs as the FP64 path (see tcorr_internal.cuh), with every operand split
// into OZ_S signed integer slices of OZ_BETA bits.
//
//   x = 2^E x',  |x'| <= 1,  x' = sum_{i=1..S} a_i 2^{-beta i} + r,  |r| <= 2^{-beta S - 1}
//
// with one power-of-two scale per operand side (E_A for G and T2K, E_B for
// T2R and AoN), so the four K segments of a group share one accumulator.  A
// slice value is an integer with |a_1| <= 2^beta and |a_i| <= 2^(beta-1)
// after that, exact in BF16.  The product of two scaled operands keeps the
// slice pairs with i + j <= S + 1:
//
//   x'y' ~ sum_{t=2..S+1} 2^{-beta t} P_t,   P_t = sum_{i+j=t} a_i b_j.
//
// Over a block of OZ_KB K chunks of 32 elements |P_t| < 2^24 (bounds below),
// so the FP32 tensor-core accumulation of P_t (a fresh TMEM accumulator per
// weight t and block) is exact: no rounding happens anywhere in the products.
// The epilogue warps convert each block's P_t to int32 (exact) and add it,
// shifted by beta (S + 1 - t) bits, into int64 running totals, exact too;
// the U element is total * 2^{E_A + E_B - beta (S + 1)} as a float-float pair.
// The error is that of representing each operand with beta S bits below its
// side's largest magnitude.  U is stored in the FP64 path's layout and the
// FP64 epilogue's float-float form does the rest.
//
// Kernel structure: SM pairs (tcgen05 cta_group::2, M = 256), the roles of the
// split-precision pair kernel (gemm_tc.cu, tc_pair.cuh).  Warp 0 loads per chunk
// the S A planes (128 pair rows of its CTA, 64-byte K rows, one box) and half of
// the S B planes (the pass's rows of a); the even CTA's warp 1 issues the
// S(S+1)/2 slice-pair MMAs into the S weight accumulators of a TMEM block of up
// to OZ_KB chunks; warps 2-9 drain and accumulate, weight by weight, the
// conversions after the weight is handed back; warp 10 decodes the items.  Every
// wait is bounded as in the split-precision kernel.
// What bounds it: operand ingest (55 KB per chunk and SM) and the MMAs.  52 tasks
// of o=40, v=300 took 98 ms on single SMs (M = 128, passes of 96 columns for any
// v, TMEM blocks of 8 chunks whose whole drain the MMAs waited for) and take 71 ms.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "tc_pair.cuh"

namespace tcorr {
namespace {

// t * 2^k as a float-float pair (hi, lo), hi + lo = t 2^k to about 2^-48
// relative, with integer and FP32 operations only: t = t2 2^48 + t1 2^24 + t0
// with |t2| < 2^15 and 0 <= t1, t0 < 2^24, each part exact in FP32; Knuth's
// TwoSum of the two largest, then the smallest added (one rounding, of the
// small parts only); the power-of-two scale is exact in the normal range.
__device__ __forceinline__ float2 int64_to_ff(long long t, int k) {
    const long long t2 = t >> 48;
    const long long rem = t - (t2 << 48);
    const float f2 = (float)(int)t2 * 0x1p48f, f1 = (float)(int)(rem >> 24) * 0x1p24f;
    const float f0 = (float)(int)(rem & 0xffffff);
    float s = f2 + f1, bb = s - f2;
    float e = (f2 - (s - bb)) + (f1 - bb);  // s + e == f2 + f1
    const float s2 = s + f0, b2 = s2 - s;
    e += (s - (s2 - b2)) + (f0 - b2);       // s2 + e == t up to the rounding of e
    const float hi = s2 + e, lo = e - (hi - s2);
    return make_float2(ldexpf(hi, k), ldexpf(lo, k));
}


using namespace tcx;

constexpr int OZ_S = 5;          // slices per operand
constexpr int OZ_BETA = 7;       // bits per slice
constexpr int OZ_N = 96;         // most a columns per item
constexpr int OZ_ROW = 64;       // K bytes per shared-memory row (32 BF16)
constexpr int OZ_A = PAIR_BM * OZ_ROW;      // 8 KB per A plane
constexpr int OZ_B = OZ_N / 2 * OZ_ROW;     // 3 KB per B plane (half of the columns per CTA)
constexpr int OZ_STAGE = OZ_S * (OZ_A + OZ_B);
constexpr int OZ_STAGES = 4;
constexpr int OZ_SMEM = OZ_STAGES * OZ_STAGE + 1024;
// One TMEM accumulator block of OZ_S weights x OZ_N columns, handed over weight
// by weight (below)
static_assert(OZ_S * OZ_N <= 512, "weight accumulators exceed the 512 TMEM columns");
static_assert(OZ_A % 1024 == 0 && OZ_B % 1024 == 0, "planes keep the 64-byte swizzle pattern aligned");
constexpr int OZ_KB = 18;        // most K chunks accumulated in TMEM per block (exact, see below)
// Exactness of a block's weight sums in FP32: |a_1| <= 2^beta, |a_i| <= 2^(beta-1)
// for i >= 2.  Weight t = i + j - 2 holds (1, 1) alone for t = 0, else (1, t+1) and
// (t+1, 1) and t - 1 pairs of two smaller factors; the largest sum is t = OZ_S - 1's.
static_assert(32LL * OZ_KB * (1 << (2 * OZ_BETA)) <= (1 << 24), "weight (1,1) must stay exact in FP32");
static_assert(32LL * OZ_KB * (2 * (1 << (2 * OZ_BETA - 1)) + (OZ_S - 2) * (1 << (2 * OZ_BETA - 2))) <= (1 << 24),
              "weight sums must stay exact in FP32");
// chunks per block: the item's nch chunks in as few blocks as exactness allows, evenly
__host__ __device__ inline int oz_block(int nch) {
    const int nblk = (nch + OZ_KB - 1) / OZ_KB;
    return (nch + nblk - 1) / nblk;
}

// The slice products of weight t (i + j = t + 2) of one K chunk into its
// accumulator (columns t * OZ_N of tmem); a0, b0: descriptor low words of the
// stage's A and B slice planes.  FIRST: the chunk opens the accumulator block,
// so the weight's first product zeroes it.
template <int T, bool FIRST>
__device__ __forceinline__ void oz_weight(uint32_t tmem, uint32_t a0, uint32_t b0, uint32_t idesc, int nks) {
    const uint32_t d = tmem + (uint32_t)(T * OZ_N);
#pragma unroll
    for (int ia = 0; ia <= T; ia++) {
        const uint32_t a = a0 + (uint32_t)((ia * OZ_A) >> 4), b = b0 + (uint32_t)(((T - ia) * OZ_B) >> 4);
        if (FIRST && ia == 0) mma_lo<2, 2, false>(d, a, b, idesc);
        else mma_lo<2, 2, true>(d, a, b, idesc);
        if (nks > 1) mma_lo<2, 2, true>(d, a + 2, b + 2, idesc);
    }
}
// one weight of a block's first chunk (waits until it is drained); false on expiry
template <int T>
__device__ __forceinline__ bool oz_open(uint32_t tmem, uint32_t a0, uint32_t b0, uint32_t idesc, int nks, uint32_t hfull0,
                                        uint32_t hempty0, uint32_t parity, bool last, volatile int *abort_flag) {
    if (!wait_warp(hempty0 + 8u * T, parity, abort_flag)) return false;
    tc_fence_after();
    if (elect_one()) {
        oz_weight<T, true>(tmem, a0, b0, idesc, nks);
        if (last) tc_commit_pair(hfull0 + 8u * T, (uint16_t)3);
    }
    __syncwarp();
    return true;
}
template <int T>
__device__ __forceinline__ void oz_next(uint32_t tmem, uint32_t a0, uint32_t b0, uint32_t idesc, int nks, uint32_t hfull0,
                                        bool last) {
    oz_weight<T, false>(tmem, a0, b0, idesc, nks);
    if (last) tc_commit_pair(hfull0 + 8u * T, (uint16_t)3);
}

__global__ void __launch_bounds__(PAIR_THREADS, 1) ugemm_oz_kernel(const __grid_constant__ Wave wv) {
    extern __shared__ __align__(1024) uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[OZ_STAGES], bar_empty[OZ_STAGES];
    __shared__ __align__(8) uint64_t bar_hfull[OZ_S], bar_hempty[OZ_S];
    __shared__ __align__(8) uint64_t bar_fin;
    __shared__ __align__(8) uint64_t bar_sfull[PAIR_SLOTS], bar_sempty[PAIR_SLOTS];
    __shared__ PairSlot slots[PAIR_SLOTS];
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank(), cid = cluster_id(), ncl = cluster_count();
    const bool leader = rank == 0;
    const uint32_t sbase = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t peer_abort = peer_addr(smem_u32((const void *)&abort_sh), rank ^ 1u);

    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_STAGES; s++) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int t = 0; t < OZ_S; t++) {
            mbar_init(smem_u32(&bar_hfull[t]), 1);
            mbar_init(smem_u32(&bar_hempty[t]), PAIR_HEMPTY_ARRIVALS);
        }
        mbar_init(smem_u32(&bar_fin), 1);
        for (int n = 0; n < PAIR_SLOTS; n++) {
            mbar_init(smem_u32(&bar_sfull[n]), 1);
            mbar_init(smem_u32(&bar_sempty[n]), (leader ? 2 : 1) + PAIR_EPI / 32);  // producer, drains, MMA issuer
        }
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
    // D = F32, A = B = BF16, K-major, M = 256 over the pair
    constexpr uint32_t idesc_m = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * PAIR_BM >> 4) << 24);

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        int last_phase[OZ_STAGES];
        for (int s = 0; s < OZ_STAGES; s++) last_phase[s] = -1;
        bool ok = true;
        bool inject = wv.inject_stall != 0 && cid == 0 && leader;
        for (uint32_t n = 0; ok; n++) {
            const PairSlot &sl = slots[n % PAIR_SLOTS];
            if (!wait_warp(smem_u32(&bar_sfull[n % PAIR_SLOTS]), (n / PAIR_SLOTS) & 1u, &abort_sh)) {
                if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_FULL);
                ok = false;
                break;
            }
            if (uni(sl.end)) break;
            const InstDesc *d = uni(sl.d);
            const int o = uni(sl.o), kv = uni(sl.kv), ko = uni(sl.ko);
            const int pp = uni(sl.p), q = uni(sl.q), cb = uni(sl.cb), cc = uni(sl.cc);
            const int s = uni(sl.box[0].x), ca = uni(sl.box[0].y);
            const uint32_t stage_tx = uni(sl.stage_tx);
            if (lane == 0) mbar_arrive(smem_u32(&bar_sempty[n % PAIR_SLOTS]));
            for (int seg = 0; seg < 4 && ok; seg++) {
                const int klen = seg < 2 ? kv : ko;
                int amap, aslice, bmap, brow;
                switch (seg) {
                    case 0: amap = MAP_G_NAT; aslice = q; bmap = MAP_T2R; brow = s * o + pp; break;
                    case 1: amap = MAP_G_SWP; aslice = pp; bmap = MAP_T2R; brow = s * o + q; break;
                    case 2: amap = MAP_T2K_NAT; aslice = pp; bmap = MAP_AON; brow = q * o + s; break;
                    default: amap = MAP_T2K_SWP; aslice = q; bmap = MAP_AON; brow = pp * o + s; break;
                }
                for (int kk = 0; kk < klen; kk++) {
                    if (!wait_warp(smem_u32(&bar_empty[stage]), phase ^ 1u, &abort_sh)) {
                        if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_EMPTY);
                        ok = false;
                        break;
                    }
                    const uint32_t full = smem_u32(&bar_full[stage]);
                    const uint32_t full_l = peer_addr(full, 0);
                    last_phase[stage] = (int)phase;
                    const uint32_t sA = sbase + stage * OZ_STAGE, sB = sA + OZ_S * OZ_A;
                    const int k0 = kk * 32;
                    if (elect_one()) {
                        if (leader) mbar_expect_tx(full, stage_tx);
                        if (!inject) {
                            // the five A planes in one box; B planes at a fixed pitch, one copy each
                            tma_load_5d_pair(sA, &d->maps[amap][0], full_l, k0, cc, cb, aslice, 0);
#pragma unroll
                            for (int pl = 0; pl < OZ_S; pl++)
                                tma_load_4d_pair(sB + pl * OZ_B, &d->maps[bmap][0], full_l, k0, ca, brow, pl);
                        }
                    }
                    __syncwarp();
                    if (inject) {
                        inject = false;
                        last_phase[stage] = -1;  // the leader's bytes never come: the MMA's wait must expire
                    }
                    if (++stage == OZ_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        }
        if (!ok && lane == 0) {
            // let the copies in flight land: the leader sees both CTAs' bytes on
            // its own full barriers; the peer gives its own copies a fixed time
            if (leader) {
                for (int s = 0; s < OZ_STAGES; s++) {
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
            uint32_t phase = 0;
            uint32_t hblk = 0;  // accumulator blocks issued
            bool ok = true;
            const uint32_t tm = uni(tmem), hfull0 = smem_u32(&bar_hfull[0]), hempty0 = smem_u32(&bar_hempty[0]);
            for (uint32_t n = 0; ok; n++) {
                const PairSlot &sl = slots[n % PAIR_SLOTS];
                if (!wait_warp(smem_u32(&bar_sfull[n % PAIR_SLOTS]), (n / PAIR_SLOTS) & 1u, &abort_sh)) {
                    if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_FULL);
                    break;
                }
                if (uni(sl.end)) break;
                const int kv = uni(sl.kv), ko = uni(sl.ko), N = uni(sl.N), nch = 2 * kv + 2 * ko;
                const int v = uni(sl.v), o = uni(sl.o);
                if (lane == 0) mbar_arrive(smem_u32(&bar_sempty[n % PAIR_SLOTS]));
                // a segment's last chunk holds one K step of data (16 values or fewer) or two
                const bool dh = v - (kv - 1) * 32 <= 16, lh = o - (ko - 1) * 32 <= 16;
                const uint32_t idesc = idesc_m | ((uint32_t)(N >> 3) << 17);
                const int kb = oz_block(nch);
                for (int c0 = 0; c0 < nch && ok; c0 += kb) {
                    const int c1 = min(c0 + kb, nch);
                    for (int ch = c0; ch < c1; ch++) {
                        if (!wait_warp(smem_u32(&bar_full[stage]), phase, &abort_sh)) {
                            if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_FULL);
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = desc_lo(sbase + stage * OZ_STAGE), b0 = a0 + (uint32_t)((OZ_S * OZ_A) >> 4);
                        const bool tail = (dh && (ch == kv - 1 || ch == 2 * kv - 1)) ||
                                          (lh && (ch == 2 * kv + ko - 1 || ch == nch - 1));
                        const int nks = tail ? 1 : 2;
                        const bool last = ch == c1 - 1;
                        // Every slice product is exact in FP32, so their order within a
                        // block is free: weight by weight.  A block's first chunk opens each
                        // weight once the drain has read it from the block before, and its
                        // last chunk hands each weight over when its products are issued, so
                        // the drain of one block overlaps the ends of both.
                        if (ch == c0) {
                            const uint32_t par = (hblk & 1u) ^ 1u;
                            ok = oz_open<0>(tm, a0, b0, idesc, nks, hfull0, hempty0, par, last, &abort_sh) &&
                                 oz_open<1>(tm, a0, b0, idesc, nks, hfull0, hempty0, par, last, &abort_sh) &&
                                 oz_open<2>(tm, a0, b0, idesc, nks, hfull0, hempty0, par, last, &abort_sh) &&
                                 oz_open<3>(tm, a0, b0, idesc, nks, hfull0, hempty0, par, last, &abort_sh) &&
                                 oz_open<4>(tm, a0, b0, idesc, nks, hfull0, hempty0, par, last, &abort_sh);
                            if (!ok) {
                                if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_TMEM);
                                break;
                            }
                            if (elect_one()) tc_commit_pair(smem_u32(&bar_empty[stage]), (uint16_t)3);
                        } else if (elect_one()) {
                            oz_next<0>(tm, a0, b0, idesc, nks, hfull0, last);
                            oz_next<1>(tm, a0, b0, idesc, nks, hfull0, last);
                            oz_next<2>(tm, a0, b0, idesc, nks, hfull0, last);
                            oz_next<3>(tm, a0, b0, idesc, nks, hfull0, last);
                            oz_next<4>(tm, a0, b0, idesc, nks, hfull0, last);
                            tc_commit_pair(smem_u32(&bar_empty[stage]), (uint16_t)3);
                        }
                        __syncwarp();
                        if (++stage == OZ_STAGES) { stage = 0; phase ^= 1u; }
                    }
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
    } else if (warp == 2 + PAIR_EPI / 32) {
        pair_scheduler(wv, cid, ncl, rank, slots, bar_sfull, bar_sempty, &abort_sh, peer_abort);
    } else {
        const int wq = warp & 3;              // TMEM lane quarter of this warp
        const int half = (warp - 2) >> 2;     // column half of each weight
        const int row = wq * 32 + lane;       // accumulator row = pair in tile
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        uint32_t hblk = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; n++) {
            const PairSlot &sl = slots[n % PAIR_SLOTS];
            if (!wait_warp(smem_u32(&bar_sfull[n % PAIR_SLOTS]), (n / PAIR_SLOTS) & 1u, &abort_sh)) {
                if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_FULL);
                break;
            }
            if (sl.end) break;
            const int nch = 2 * (sl.kv + sl.ko), kb = oz_block(nch), nhb = (nch + kb - 1) / kb;
            const int hw = sl.N / 2;          // columns of this warp, a multiple of 8
            long long tot[OZ_N / 2];
#pragma unroll
            for (int j = 0; j < OZ_N / 2; j++) tot[j] = 0;
            for (int hb = 0; hb < nhb && ok; hb++) {
#pragma unroll
                for (int t = 0; t < OZ_S; t++) {
                    if (ok) {
                        ok = wait_warp(smem_u32(&bar_hfull[t]), hblk & 1u, &abort_sh);
                        if (ok) {
                            // the weight is free once its columns are in registers: the
                            // conversions run beside the next block's products
                            const long long wgt = 1LL << (OZ_BETA * (OZ_S - 1 - t));
                            uint32_t r[OZ_N / 16][8];
                            tc_fence_after();
#pragma unroll
                            for (int c8 = 0; c8 < OZ_N / 16; c8++)
                                if (c8 * 8 < hw)
                                    tc_ld8(tmem + lane_off + (uint32_t)(t * OZ_N + half * hw + c8 * 8), r[c8]);
                            tc_wait_ld();
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive_cluster(peer_addr(smem_u32(&bar_hempty[t]), 0));
#pragma unroll
                            for (int c8 = 0; c8 < OZ_N / 16; c8++)
                                if (c8 * 8 < hw) {
#pragma unroll
                                    for (int j = 0; j < 8; j++)
                                        tot[c8 * 8 + j] += (long long)__float2int_rn(__uint_as_float(r[c8][j])) * wgt;
                                }
                        }
                    }
                }
                hblk++;
            }
            if (!ok) {
                if (lane == 0) fail_pair(&abort_sh, peer_abort, wv.err, DERR_TIMEOUT_TMEM);
                break;
            }
            // U^g[a][b][c] in the FP64 path's layout, each value as a float-float
            // (hi, lo) pair in its 8 bytes (about 48 significant bits), so that the
            // epilogue works on the FP32 pipe; formed from the exact int64 total
            // without the FP64 pipe (int64_to_ff)
            const int v = sl.v, pc = sl.pc, vc = round_up(v, UPAD);
            const int b = sl.cb + row / pc, c = sl.cc + row % pc;
            if (!sl.empty && b < v && c < v) {
                const int scale_exp = sl.scale - OZ_BETA * (OZ_S + 1);
                const int a0 = sl.pass0 + half * hw;
                const int64_t stride = (int64_t)v * vc;
                // One branch past eight columns: at small v an item is so short that
                // fetching the instructions of this part bounds it, and a branch past
                // every column cost as much as the column (contraction of o=30: v=17
                // 6.12 ms with those, 3.32 so; v=33 18.0 and 10.3; o=12: v=48 1.00 and
                // 0.85, v=72 3.37 and 3.34; 52 tasks of o=40, v=300 70.66 both.  A
                // multiplication by two powers of two in place of ldexpf gave no more
                // and made the last 71.0; a loop over the weights that is not unrolled
                // is 5% slower from v=72 on).
                float2 *Ug = static_cast<float2 *>(wv.U) + sl.u_off + (int64_t)sl.g * (sl.ug3 / 3) + (int64_t)b * vc + c +
                             (int64_t)a0 * stride;
#pragma unroll
                for (int c8 = 0; c8 < OZ_N / 16; c8++)
                    if (c8 * 8 < hw && a0 + c8 * 8 < v) {
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            if (a0 + c8 * 8 + j < v) *Ug = int64_to_ff(tot[c8 * 8 + j], scale_exp);
                            Ug += stride;
                        }
                    }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_sempty[n % PAIR_SLOTS]));
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

// ---- scales ------------------------------------------------------------------------
// Max |x| over n doubles: non-negative doubles order like their bit patterns.
__global__ void maxabs_kernel(const double *__restrict__ x, int64_t n, unsigned long long *out) {
    unsigned long long m = 0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned long long)__double_as_longlong(fabs(x[k])));
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Scale exponents: e[0] for the A side (max of vvvo and t2), e[1] for the B
// side (max of t2 and ooov): the smallest E with max |x| <= 2^E.
__global__ void oz_exponents_kernel(const unsigned long long *m, int *e) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const double a = fmax(__longlong_as_double((long long)m[0]), __longlong_as_double((long long)m[1]));
    const double b = fmax(__longlong_as_double((long long)m[1]), __longlong_as_double((long long)m[2]));
    int ea = 0, eb = 0;
    // infinite or NaN: any exponent, the energies are NaN (eps_ff_kernel)
    if (a > 0.0 && isfinite(a)) frexp(a, &ea);  // a = f 2^ea, f in [0.5, 1): a < 2^ea
    if (b > 0.0 && isfinite(b)) frexp(b, &eb);
    e[0] = ea;
    e[1] = eb;
}
__global__ void seed_max_kernel(unsigned long long *m, double x) {
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicMax(m, (unsigned long long)__double_as_longlong(fabs(x)));
}

}  // namespace

int oz_slices() { return OZ_S; }

cudaError_t launch_maxabs(const double *x, int64_t n, unsigned long long *out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 2048);
    maxabs_kernel<<<(unsigned)blocks, 256, 0, st>>>(x, n, out);
    return cudaGetLastError();
}

cudaError_t launch_oz_exponents(const unsigned long long *m, int *e, cudaStream_t st) {
    oz_exponents_kernel<<<1, 32, 0, st>>>(m, e);
    return cudaGetLastError();
}

cudaError_t launch_seed_max(unsigned long long *m, double x, cudaStream_t st) {
    seed_max_kernel<<<1, 32, 0, st>>>(m, x);
    return cudaGetLastError();
}

cudaError_t oz_fill_desc(InstDesc &d, const Operands &op, const int *exps, std::string &err) {
    const int o = d.dm.o, v = d.dm.v, dp = d.dm.dp, lp = d.dm.lp;
    const uint64_t eb = 2;
    const CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const int pb = 8, pc = 16;  // 128 pair rows
    d.pb = pb;
    d.pc = pc;
    d.kb = 1;
    d.nbt = (v + pb - 1) / pb;
    d.nct = (v + pc - 1) / pc;
    d.pair = 1;
    d.tblk = pair_task_block(v, dp, OZ_S * eb);
    // passes of equal width, a multiple of 16: each CTA holds half of the columns
    d.npass = (v + OZ_N - 1) / OZ_N;
    d.brows = round_up((v + d.npass - 1) / d.npass, 16);
    d.kv = (v + 31) / 32;
    d.ko = (o + 31) / 32;
    d.stage_tx = (uint32_t)(2 * OZ_S * (OZ_A + d.brows / 2 * OZ_ROW));  // both CTAs' bytes
    d.oz_e = exps;
    const uint64_t V = v, O = o, S = OZ_S;
    // plane strides (bytes): one slice plane of each operand layout
    const uint64_t pG = (uint64_t)O * V * V * dp * eb, pT2K = (uint64_t)O * V * V * lp * eb;
    const uint64_t pT2R = (uint64_t)O * O * V * dp * eb, pAoN = (uint64_t)O * O * V * lp * eb;
    const uint32_t bk = 32, bpc = (uint32_t)pc, bpb = (uint32_t)pb, bn = (uint32_t)(d.brows / 2), bs = OZ_S;
    {
        uint64_t dims[5] = {V, V, V, O, S};
        uint64_t st[4] = {dp * eb, V * dp * eb, V * V * dp * eb, pG};
        uint32_t box[5] = {bk, bpc, bpb, 1, bs};
        if (!encode(&d.maps[MAP_G_NAT][0], dt, 5, op.G, dims, st, box, err, "G slices")) return cudaErrorInvalidValue;
        uint64_t st2[4] = {V * dp * eb, dp * eb, V * V * dp * eb, pG};
        if (!encode(&d.maps[MAP_G_SWP][0], dt, 5, op.G, dims, st2, box, err, "G slices swapped"))
            return cudaErrorInvalidValue;
    }
    {
        uint64_t dims[5] = {O, V, V, O, S};
        uint64_t st[4] = {lp * eb, V * lp * eb, V * V * lp * eb, pT2K};
        uint32_t box[5] = {bk, bpc, bpb, 1, bs};
        if (!encode(&d.maps[MAP_T2K_NAT][0], dt, 5, op.T2K, dims, st, box, err, "T2K slices"))
            return cudaErrorInvalidValue;
        uint64_t st2[4] = {V * lp * eb, lp * eb, V * V * lp * eb, pT2K};
        if (!encode(&d.maps[MAP_T2K_SWP][0], dt, 5, op.T2K, dims, st2, box, err, "T2K slices swapped"))
            return cudaErrorInvalidValue;
    }
    {
        uint64_t dims[4] = {V, V, O * O, S};
        uint64_t st[3] = {dp * eb, V * dp * eb, pT2R};
        uint32_t box[4] = {bk, bn, 1, 1};
        if (!encode(&d.maps[MAP_T2R][0], dt, 4, op.T2R, dims, st, box, err, "T2R slices")) return cudaErrorInvalidValue;
    }
    {
        uint64_t dims[4] = {O, V, O * O, S};
        uint64_t st[3] = {lp * eb, V * lp * eb, pAoN};
        uint32_t box[4] = {bk, bn, 1, 1};
        if (!encode(&d.maps[MAP_AON][0], dt, 4, op.AoN, dims, st, box, err, "AoN slices")) return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

int64_t oz_units_per_task(const InstDesc &d) { return (int64_t)3 * ((d.nbt * d.nct + 1) / 2) * d.npass; }

cudaError_t oz_prepare() {
    static std::mutex mu;
    static bool done = false;
    std::lock_guard<std::mutex> lk(mu);
    if (done) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(ugemm_oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
    if (e == cudaSuccess) done = true;
    return e;
}

cudaError_t launch_ugemm_oz(int sm_count, const Wave &w, cudaStream_t st) {
    if (w.n_gemm <= 0) return cudaSuccess;
    const cudaError_t e = oz_prepare();
    if (e != cudaSuccess) return e;
    static PairLaunch pl;
    return pl.launch(ugemm_oz_kernel, PAIR_THREADS, OZ_SMEM, sm_count, w.n_gemm, st, w);
}

}  // namespace tcorr
