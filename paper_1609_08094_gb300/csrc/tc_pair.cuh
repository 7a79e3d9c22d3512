// Device code shared by the SM-pair contractions (split precision and FP64
// emulation): thread-block clusters of two CTAs, one per SM of an SM pair, whose
// even CTA issues tcgen05 cta_group::2 MMAs for both.  The item decode, the
// scheduler warp that runs it ahead of the other roles, and the launch.
#pragma once

#include <algorithm>
#include <mutex>

#include "tc_common.cuh"

namespace tcorr {
namespace tcx {

constexpr int PAIR_EPI = 256;             // drain threads: warps 2-9
constexpr int PAIR_THREADS = 64 + PAIR_EPI + 32;  // warp 0: TMA producer, 1: MMA issuer, 10: scheduler
constexpr int PAIR_HEMPTY_ARRIVALS = 2 * (PAIR_EPI / 32);  // the drain warps of both CTAs
constexpr int PAIR_BM = 128;              // pair rows per CTA tile
constexpr int PAIR_BN = 256;              // widest pass
constexpr int PAIR_ROW = 128;             // one K block (two chunks) per shared-memory row, 128-byte swizzle
constexpr int PAIR_A = PAIR_BM * PAIR_ROW;  // 16 KB per A plane
// B rows of packed columns come in boxes of 16, 32, 64 or 128 rows, each within one
// entry: as few as its columns allow.  With boxes of 16 rows only, eight per plane and
// stage, the contraction of o=13, v=131 took 9.31 ms (9.01 so), of 24 molecules of
// v = 20..120 17.4 ms (17.0).
constexpr int PACK_ROWS = 16;
constexpr int PACK_BOXES = PAIR_BN / 2 / PACK_ROWS;  // most boxes per CTA and plane

struct PairCache {
    SegCache s;
    const PackRun *runs;
    const PackEnt *ents;
    int nrun, r, r_end;  // cached run and the unit after its last
    int ntb, tblk;       // tasks of the segment, and of a block
    PackRun run;
};
__device__ __forceinline__ void pair_reset(PairCache &c) { seg_reset(c.s); }
struct PairItem {
    int bt, ct;          // this CTA's pair tile
    int p, q;            // the A side's slices
    int N;               // columns of the MMAs
    int pass0, ncol;     // first column (of a, or of the run's packed columns) and valid columns
    int tb, g, s;        // not packed: task of the segment, group and its s
    int ent0;            // packed: first entry of the run
    bool packed;         // entries of a run
    bool boxes;          // several entries: B in 16-row boxes
    bool empty;          // this CTA's tile index lies past the group's tile list
    bool diag;           // i = j = k: no work
};
__device__ __forceinline__ PairItem decode_pair(const Wave &w, int64_t it, PairCache &c, uint32_t rank) {
    const bool fresh = c.s.si < 0 || it >= c.s.end;
    seg_update(w, it, c.s);
    PairItem r;
    const InstDesc &d = *c.s.d;
    const int npt = c.s.nbt * c.s.nct;
    const int npair = (npt + 1) / 2;
    int tp;
    if (fresh) {
        const Seg &sg = w.segs[c.s.si];
        c.runs = sg.runs;
        c.ents = sg.ents;
        c.nrun = sg.nrun;
        c.ntb = sg.ntb;
        const int nblk = (c.ntb + d.tblk - 1) / d.tblk;
        c.tblk = (c.ntb + nblk - 1) / nblk;  // equal blocks
        c.r = 0;
        c.r_end = -1;
    }
    r.packed = c.nrun != 0;
    r.boxes = false;
    if (r.packed) {
        const int x = (int)(it - c.s.begin);
        if (x >= c.r_end) {  // units only grow: search forward
            int lo = c.r, hi = c.nrun - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (c.runs[mid].unit0 <= x) lo = mid; else hi = mid - 1;
            }
            c.r = lo;
            c.run = c.runs[lo];
            c.r_end = c.run.unit0 + npair * c.run.npass;
        }
        const int local = x - c.run.unit0, n = local % c.run.npass;
        tp = local / c.run.npass;
        r.boxes = c.run.nent > 1;
        if (r.boxes) {
            const int cols = c.run.nent * d.packw;
            const int width = ((cols + c.run.npass - 1) / c.run.npass + 31) / 32 * 32;
            r.pass0 = n * width;
            r.ncol = min(width, cols - r.pass0);
            r.N = (r.ncol + 31) / 32 * 32;
        } else {  // v <= 256: one pass
            r.pass0 = 0;
            r.ncol = d.dm.v;
            r.N = (r.ncol + 15) / 16 * 16;
        }
        r.ent0 = c.run.ent0;
        r.p = c.run.p;
        r.q = c.run.q;
        r.tb = r.g = r.s = 0;
        r.diag = false;  // the tables hold no group of a task i = j = k
    } else {
        // N pass fastest, then group, then the tasks of a block, then tile pair: the
        // tasks of a block are neighbours (i, j, k), (i, j, k + 1), ..., whose groups
        // read the same tiles of G[i] and G[j] (two groups of a task also of G[k]),
        // and the block's rows of B stay in L2 (pair_task_block)
        const int64_t x = it - c.s.begin;
        const int per = 3 * c.s.npass;  // items of a task at one tile pair
        const int64_t blk = x / ((int64_t)per * npair * c.tblk);
        const int nt = (int)min((int64_t)c.tblk, c.ntb - blk * c.tblk);
        const int l = (int)(x - blk * c.tblk * npair * per);
        tp = l / (nt * per);
        int y = l - tp * nt * per;
        const int n = y % c.s.npass;
        y /= c.s.npass;
        r.g = y % 3;
        r.tb = (int)(blk * c.tblk) + y / 3;
        if (r.tb != c.s.tcached) {
            const int *tk = d.tasks + 3 * (c.s.task0 + r.tb);
            c.s.ti = tk[0];
            c.s.tj = tk[1];
            c.s.tk = tk[2];
            c.s.tcached = r.tb;
        }
        const int i = c.s.ti, j = c.s.tj, k = c.s.tk;
        r.diag = (i == j && j == k);
        r.s = r.g == 0 ? i : (r.g == 1 ? j : k);
        r.p = r.g == 0 ? j : i;
        r.q = r.g == 2 ? j : k;
        r.pass0 = n * d.brows;
        r.ncol = min(d.brows, d.dm.v - r.pass0);
        r.N = (r.ncol + 15) / 16 * 16;
        r.ent0 = 0;
    }
    const int t = tp * 2 + (int)rank;
    r.empty = t >= npt;
    r.bt = r.empty ? c.s.nbt : t / c.s.nct;  // past the list: b >= v, all TMA fill
    r.ct = r.empty ? 0 : t % c.s.nct;
    return r;
}
// What the roles of a CTA need of an item, written by its scheduler warp.
struct PairSlot {
    const InstDesc *d;
    int64_t u_off, ug3;     // U elements before the segment (packed) or the task, and per task
    int end;                // no more items
    int o, v, kv, ko, kind;
    int p, q, N, cb, cc;    // A slices, columns, first b and c of this CTA's tile
    uint32_t stage_tx;      // bytes of a stage, both CTAs'
    int nbx, boxes;         // B copies per plane and stage; in boxes of packed columns?
    int pc, packed, empty;
    int g, pass0, ncol;     // not packed: group and columns of a
    int scale;              // FP64 emulation: E_A + E_B
    int4 box[PACK_BOXES];   // B copies: s (-1 past the valid columns), first a, log2(rows / 16), first row
    int2 ent[PAIR_BN / 8];  // packed: (tbg, a) of columns 8 k .. 8 k + 7, a = 2^20 for none
};
constexpr int PAIR_SLOTS = 4;
// abort both CTAs of the pair and raise the device error flag
__device__ __forceinline__ void fail_pair(volatile int *abort_flag, uint32_t peer_abort_cl, int *err, int code) {
    *abort_flag = 1;
    st_cluster_u32(peer_abort_cl, 1u);
    atomicOr(err, code);
}
__device__ __forceinline__ void spin_ns(uint64_t ns) {
    const uint64_t t0 = gtimer();
    while (gtimer() - t0 < ns) {
    }
}


// Scheduler warp: decodes this CTA's items ahead of the other roles, which would
// otherwise each decode them between two items (integer divisions and dependent
// loads; ~800 clocks per item and role).
__device__ __forceinline__ void pair_scheduler(const Wave &wv, uint32_t cid, uint32_t ncl, uint32_t rank,
                                               PairSlot *slots, uint64_t *bar_sfull, uint64_t *bar_sempty,
                                               volatile int *abort_flag, uint32_t peer_abort) {
    const int lane = threadIdx.x & 31;
    PairCache pc;
    pair_reset(pc);
    uint32_t n = 0;
    bool ok = true;
    for (int64_t it = cid; ok; it += ncl) {
        const bool end = it >= wv.n_gemm;
        PairItem w;
        if (!end) {
            w = decode_pair(wv, it, pc, rank);
            if (w.diag) continue;
        }
        PairSlot &sl = slots[n % PAIR_SLOTS];
        if (n >= PAIR_SLOTS &&
            !wait_warp(smem_u32(&bar_sempty[n % PAIR_SLOTS]), (n / PAIR_SLOTS - 1) & 1u, abort_flag)) {
            if (lane == 0) fail_pair(abort_flag, peer_abort, wv.err, DERR_TIMEOUT_EMPTY);
            ok = false;
            break;
        }
        if (!end) {
            const InstDesc &d = *pc.s.d;
            if (lane == 0) {
                sl.d = &d;
                sl.ug3 = 3 * d.dm.ug;
                sl.u_off = pc.s.u_off + w.tb * (3 * d.dm.ug);
                sl.o = d.dm.o;
                sl.v = d.dm.v;
                sl.kv = d.kv;
                sl.ko = d.ko;
                sl.kind = d.kind;
                sl.p = w.p;
                sl.q = w.q;
                sl.N = w.N;
                sl.cb = w.bt * d.pb;
                sl.cc = w.ct * d.pc;
                sl.stage_tx = w.boxes ? 2u * (2u * PAIR_A + 2u * (uint32_t)(w.N / 2) * PAIR_ROW) : d.stage_tx;
                sl.boxes = w.boxes;
                sl.pc = d.pc;
                sl.packed = w.packed;
                sl.empty = w.empty;
                sl.g = w.g;
                sl.pass0 = w.pass0;
                sl.ncol = w.ncol;
                sl.scale = d.oz_e ? d.oz_e[0] + d.oz_e[1] : 0;
            }
            if (lane == 0) {
                int nbx = 1;
                if (!w.boxes) {
                    sl.box[0] = make_int4(w.packed ? pc.ents[w.ent0].s : w.s, w.pass0 + (int)rank * (w.N / 2), 0, 0);
                } else {
                    // the CTA's half of the pass, entry by entry, in the largest boxes that fit
                    const int half = w.N / 2;
                    nbx = 0;
                    for (int row = 0; row < half;) {
                        const int x = (int)rank * half + row;
                        int len = half - row, a = 0, s = -1;
                        if (x < w.ncol) {
                            const int col = w.pass0 + x, m = col / d.packw;
                            a = col - m * d.packw;
                            s = pc.ents[w.ent0 + m].s;
                            len = min(len, min(d.packw - a, w.ncol - x));
                        }
                        const int h = len >= 128 ? 3 : (len >= 64 ? 2 : (len >= 32 ? 1 : 0));
                        sl.box[nbx++] = make_int4(s, a, h, row);
                        row += PACK_ROWS << h;
                    }
                }
                sl.nbx = nbx;
            }
            if (w.packed) {
                int2 e = make_int2(0, 1 << 20);
                if (8 * lane < w.ncol) {
                    const int col = w.pass0 + 8 * lane, m = col / d.packw;
                    e = make_int2(pc.ents[w.ent0 + m].tbg, col - m * d.packw);
                }
                sl.ent[lane] = e;
            }
        }
        if (lane == 0) sl.end = end;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_sfull[n % PAIR_SLOTS]));
        if (end) break;
        n++;
    }
}

// Tasks per block of the item order: so many that the rows of T2R they read
// (four blocks [v][dp] per task that its neighbours do not) take at most 40 MB of
// the 126 MB L2, which A and U stream through.
inline int pair_task_block(int v, int dp, size_t bytes_per_value) {
    const int64_t per_task = 4 * (int64_t)v * dp * (int64_t)bytes_per_value;
    return (int)std::max<int64_t>(1, std::min<int64_t>(64, ((int64_t)40 << 20) / per_task));
}

// Launch of a pair kernel on as many 2-CTA clusters as are co-resident (one
// per SM pair that the cluster scheduler can place), queried once per device.
struct PairLaunch {
    std::mutex mu;
    int cache[64] = {};
    template <typename K, typename... A>
    cudaError_t launch(K kernel, int threads, int smem, int sm_count, int64_t items, cudaStream_t st, const A &...args) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(sm_count / 2 * 2), 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)smem;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int dev = 0, n = sm_count / 2;
        if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
            std::lock_guard<std::mutex> lk(mu);
            if (cache[dev] == 0) {
                int m = 0;
                if (cudaOccupancyMaxActiveClusters(&m, kernel, &cfg) != cudaSuccess || m < 1) {
                    cudaGetLastError();
                    m = sm_count / 2;
                }
                cache[dev] = std::min(m, sm_count / 2);
            }
            n = cache[dev];
        }
        cfg.gridDim = dim3((unsigned)(2 * std::min<int64_t>(n, items)), 1, 1);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
};

}  // namespace tcx
}  // namespace tcorr
