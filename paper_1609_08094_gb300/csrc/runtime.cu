// Host runtime shared by the C ABI front ends: see runtime.cuh.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <limits>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <tuple>
#include <vector>

#include "runtime.cuh"

namespace tcorr {
namespace rt {

thread_local std::string g_create_error;

// Handles that come and go (one per molecule) spent most of their time in
// cudaMalloc, cudaFree and the pinned allocations: o=10, v=100 in BF16X3 took 0.83
// ms to create and 2.65 ms to destroy around 2.1 ms of work.  Their device
// allocations of up to POOL_MAX bytes come from one stream-ordered pool per device
// that keeps at most POOL_KEEP bytes when they are gone; of the larger ones, from
// cudaMalloc, up to LIST_KEEP bytes per device are kept for a later handle that
// asks for as much or up to a fifth less, the oldest given back first.  Both are
// given back when an allocation of a handle or a server fails, when a server is
// created, and by tcorr_trim; another user of the device has the latter.  The two
// bounds are 4 GiB together, 1.5% of the device: a U scratch above 3.5 GiB (up to
// 16 GiB) goes back when its handle is closed, as all did before.  (Growing the pool by the gigabytes of a U
// scratch took 2 ms more than cudaMalloc: o=12, v=82 took 2.8 ms to create and 4.0
// to destroy while earlier handles were alive, 0.8 and 2.4 with cudaMalloc alone.)
// Pinned blocks of up to 1 MiB are kept for reuse, at most 32 of them.  Pool and
// lists are safe with several threads; a block enters a list after its handle's
// stream has been synchronised.
constexpr size_t POOL_MAX = (size_t)16 << 20, POOL_KEEP = (size_t)512 << 20, LIST_KEEP = (size_t)3584 << 20;
namespace {
struct DevList {
    std::mutex mu;
    std::vector<Exec::DevPtr> blocks;  // oldest first
    size_t kept = 0;
};
DevList &dev_list(int dev) {
    static DevList *l = new DevList[64];  // outlives every handle
    return l[dev];
}
// Gives back the oldest blocks until at most `keep` bytes are kept
void trim_list(DevList &l, size_t keep) {
    for (;;) {
        Exec::DevPtr d;
        {
            std::lock_guard<std::mutex> lk(l.mu);
            if (l.kept <= keep) return;
            d = l.blocks.front();
            l.kept -= d.bytes;
            l.blocks.erase(l.blocks.begin());
        }
        cudaFree(d.p);
    }
}
// The smallest kept block of at least `bytes` and at most a quarter more
bool take_kept(DevList &l, size_t bytes, Exec::DevPtr &d) {
    std::lock_guard<std::mutex> lk(l.mu);
    l.blocks.reserve(LIST_KEEP / POOL_MAX + 1);  // giving a block back must not allocate (dev_free)
    size_t best = l.blocks.size();
    for (size_t n = 0; n < l.blocks.size(); n++)
        if (l.blocks[n].bytes >= bytes && l.blocks[n].bytes - bytes <= bytes / 4 &&
            (best == l.blocks.size() || l.blocks[n].bytes < l.blocks[best].bytes))
            best = n;
    if (best == l.blocks.size()) return false;
    d = l.blocks[best];
    l.kept -= d.bytes;
    l.blocks.erase(l.blocks.begin() + best);
    return true;
}
}  // namespace
namespace {
struct Pools {
    std::mutex mu;
    cudaMemPool_t p[64] = {};
};
Pools &pools() {
    static Pools *l = new Pools();
    return *l;
}
}  // namespace
static cudaMemPool_t handle_pool(int dev) {
    if (dev < 0 || dev >= 64) return nullptr;
    Pools &l = pools();
    std::lock_guard<std::mutex> lk(l.mu);
    if (!l.p[dev]) {
        cudaMemPoolProps pp{};
        pp.allocType = cudaMemAllocationTypePinned;
        pp.location.type = cudaMemLocationTypeDevice;
        pp.location.id = dev;
        cudaMemPool_t p = nullptr;
        uint64_t keep = POOL_KEEP;
        if (cudaMemPoolCreate(&p, &pp) != cudaSuccess ||
            cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;  // plain cudaMalloc instead
        }
        l.p[dev] = p;
    }
    return l.p[dev];
}

void give_back_kept(int dev) {
    if (dev < 0 || dev >= 64) return;
    trim_list(dev_list(dev), 0);
    Pools &l = pools();
    std::lock_guard<std::mutex> lk(l.mu);
    if (l.p[dev]) cudaMemPoolTrimTo(l.p[dev], 0);
}

// Room for one more element: what is noted after an allocation cannot fail then
template <typename T>
static void reserve_one(std::vector<T> &v) {
    if (v.size() == v.capacity()) v.reserve(2 * v.size() + 16);
}

void *dalloc_bytes(Exec &ex, size_t bytes) {
    if (bytes == 0) bytes = 16;
    const bool handle = ex.pool && ex.pool_max != SIZE_MAX;
    reserve_one(ex.dev);
    Exec::DevPtr d{nullptr, bytes, ex.pool && bytes <= ex.pool_max, handle && bytes > ex.pool_max};
    cudaError_t e = cudaSuccess;
    if (!d.listed || !take_kept(dev_list(ex.device), bytes, d))
        for (int rep = 0; rep < 2; rep++) {
            e = d.pooled ? cudaMallocFromPoolAsync(&d.p, bytes, ex.pool, ex.stream) : cudaMalloc(&d.p, bytes);
            if (e == cudaSuccess) break;
            cudaGetLastError();
            give_back_kept(ex.device);  // then once more, the server's allocations too
        }
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw Fail{TCORR_ENOMEM, "cudaMalloc of " + std::to_string(bytes) + " bytes failed: " +
                                     cudaGetErrorString(e)};
    }
    ex.dev.push_back(d);
    ex.bytes += d.bytes;  // of a kept block its size, up to a quarter more than asked for
    return d.p;
}

void copy_in(Exec &ex, void *dst, const void *src, size_t bytes) {
    if (bytes == 0) return;
    const unsigned char *p = static_cast<const unsigned char *>(src);
    ex.sources.emplace_back(p, p + bytes);
    CK(cudaMemcpyAsync(dst, ex.sources.back().data(), bytes, cudaMemcpyHostToDevice, ex.stream));
}
void copied_in(Exec &ex) { ex.sources.clear(); }

static void dev_free(Exec &ex, const Exec::DevPtr &d) {
    if (d.listed && d.bytes <= LIST_KEEP && cudaStreamSynchronize(ex.stream) == cudaSuccess) {
        DevList &l = dev_list(ex.device);
        trim_list(l, LIST_KEEP - d.bytes);
        std::lock_guard<std::mutex> lk(l.mu);
        if (l.kept + d.bytes <= LIST_KEEP) {  // another thread may have filled it
            l.blocks.push_back(d);
            l.kept += d.bytes;
            return;
        }
    }
    if (!d.pooled || cudaFreeAsync(d.p, ex.stream) != cudaSuccess) cudaFree(d.p);
}

void dfree(Exec &ex, void *p) {
    if (!p) return;
    for (size_t n = 0; n < ex.dev.size(); n++)
        if (ex.dev[n].p == p) {
            ex.bytes -= ex.dev[n].bytes;
            dev_free(ex, ex.dev[n]);
            ex.dev.erase(ex.dev.begin() + n);
            return;
        }
}

size_t free_device_bytes(const Exec &ex) {
    size_t free_b = 0, total_b = 0;
    CK(cudaMemGetInfo(&free_b, &total_b));
    if (ex.pool) {
        uint64_t reserved = 0, used = 0;
        if (cudaMemPoolGetAttribute(ex.pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
            cudaMemPoolGetAttribute(ex.pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess && reserved > used)
            free_b += reserved - used;
        if (ex.pool_max != SIZE_MAX) {
            DevList &l = dev_list(ex.device);
            std::lock_guard<std::mutex> lk(l.mu);
            free_b += l.kept;
        }
    }
    return free_b;
}

// Pinned blocks kept for reuse
namespace {
struct PinList {
    std::mutex mu;
    std::vector<Exec::HostPtr> blocks;
};
PinList &pin_list() {
    static PinList *l = new PinList();  // outlives every handle
    return *l;
}
constexpr size_t PIN_UNIT = (size_t)64 << 10, PIN_MAX = (size_t)1 << 20, PIN_BLOCKS = 32;
}  // namespace

void *halloc_bytes(Exec &ex, size_t bytes) {
    bytes = std::max<size_t>(1, (bytes + PIN_UNIT - 1) / PIN_UNIT) * PIN_UNIT;
    Exec::HostPtr h{nullptr, bytes};
    reserve_one(ex.host);
    if (bytes <= PIN_MAX) {
        PinList &l = pin_list();
        std::lock_guard<std::mutex> lk(l.mu);
        l.blocks.reserve(PIN_BLOCKS);  // giving a block back must not allocate (host_free)
        for (size_t n = 0; n < l.blocks.size(); n++)
            if (l.blocks[n].bytes == bytes) {
                h = l.blocks[n];
                l.blocks.erase(l.blocks.begin() + n);
                break;
            }
    }
    if (!h.p) CK(cudaHostAlloc(&h.p, bytes, cudaHostAllocPortable));
    ex.host.push_back(h);
    return h.p;
}

void give_back_pinned() {
    PinList &l = pin_list();
    for (;;) {
        Exec::HostPtr h;
        {
            std::lock_guard<std::mutex> lk(l.mu);
            if (l.blocks.empty()) return;
            h = l.blocks.back();
            l.blocks.pop_back();
        }
        cudaFreeHost(h.p);
    }
}

static void host_free(const Exec::HostPtr &h) {
    if (h.bytes <= PIN_MAX) {
        PinList &l = pin_list();
        std::lock_guard<std::mutex> lk(l.mu);
        if (l.blocks.size() < PIN_BLOCKS) {
            l.blocks.push_back(h);
            return;
        }
    }
    cudaFreeHost(h.p);
}

void hfree(Exec &ex, void *p) {
    if (!p) return;
    for (size_t n = 0; n < ex.host.size(); n++)
        if (ex.host[n].p == p) {
            host_free(ex.host[n]);
            ex.host.erase(ex.host.begin() + n);
            return;
        }
}

// The caller has synchronised ex.stream (or, in the server's stream order, its
// pool's frees run after the work)
void release(Exec &ex) {
    for (const Exec::DevPtr &d : ex.dev) dev_free(ex, d);
    ex.bytes = 0;
    for (const Exec::HostPtr &h : ex.host) host_free(h);
    for (auto &pe : ex.pending) {
        cudaEventDestroy(pe.a);
        cudaEventDestroy(pe.b);
    }
    const bool any = !ex.dev.empty();
    ex.dev.clear();
    ex.host.clear();
    ex.pending.clear();
    if (any && ex.pool && ex.pool_max != SIZE_MAX) {  // a handle: give back what is above the bound
        uint64_t reserved = 0;
        if (cudaMemPoolGetAttribute(ex.pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
            reserved > POOL_KEEP) {
            cudaStreamSynchronize(ex.stream);
            cudaMemPoolTrimTo(ex.pool, POOL_KEEP);
        }
    }
}

// Copy (or reference) one caller array on the device.  For host inputs the
// data is staged into a temporary device buffer that free_tmp releases.
const double *device_view(Exec &ex, const double *src, size_t n, bool host, double *&tmp) {
    tmp = nullptr;
    if (!host) return src;
    dalloc(ex, tmp, n * sizeof(double));
    CK(cudaMemcpyAsync(tmp, src, n * sizeof(double), cudaMemcpyHostToDevice, ex.stream));
    return tmp;
}

void free_tmp(Exec &ex, double *&tmp) {
    if (!tmp) return;
    CK(cudaStreamSynchronize(ex.stream));
    dfree(ex, tmp);
    tmp = nullptr;
}

// Accumulate the recorded event pairs; call after a stream synchronisation.
void resolve_timers(Exec &ex) {
    std::vector<Exec::Pending> keep;
    for (auto &pe : ex.pending) {
        if (cudaEventQuery(pe.b) == cudaErrorNotReady) {  // still in flight: keep for later
            keep.push_back(pe);
            continue;
        }
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, pe.a, pe.b) == cudaSuccess) {
            ex.k_ms[pe.cls] += ms;
            ex.k_launch[pe.cls] += 1;
        }
        cudaEventDestroy(pe.a);
        cudaEventDestroy(pe.b);
    }
    cudaGetLastError();
    ex.pending.swap(keep);
}

double problem_flops(int o, int v) {
    const double tasks = (double)o * (o + 1) * (o + 2) / 6.0 - o;  // i = j = k tasks carry no work
    return tasks * 12.0 * (double)v * v * v * (double)(v + o);
}

int operand_prec(int prec, int o, int v) {
    if (prec == TCORR_BF16X3 && problem_flops(o, v) < BF16_MIN_FLOPS) return TCORR_TF32X3;
    return prec;
}

int elem_kind(int prec) { return prec == TCORR_FP64 ? 0 : (prec == TCORR_TF32X3 ? 1 : (prec == TCORR_BF16X3 ? 2 : 3)); }
bool is_split(int prec) { return prec == TCORR_TF32X3 || prec == TCORR_BF16X3; }
bool fp64_epilogue(int prec) { return prec == TCORR_FP64 || prec == TCORR_FP64_OZ; }
size_t elem_bytes(int prec) { return prec == TCORR_FP64 ? 8 : (prec == TCORR_TF32X3 ? 4 : 2); }
size_t u_elem_bytes(int prec) { return fp64_epilogue(prec) ? 8 : 4; }
// operand planes per element: 1 (FP64), 2 (hi + lo), or the FP64-emulation slices
static size_t operand_planes(int prec) { return prec == TCORR_FP64 ? 1 : (is_split(prec) ? 2 : (size_t)oz_slices()); }

// Streams a host array of v rows of `row` doubles to the device in chunks of
// up to 512 MB and calls consume(stage, d0, nr) for each, which enqueues the
// chunk's kernels on ex.stream.  Two staging buffers and a copy stream of
// its own: the copy of chunk n+1 overlaps the kernels of chunk n (the host
// array should be pinned for the copies to run asynchronously).
struct CopyPipe {
    cudaStream_t cs = nullptr;
    cudaEvent_t ev[5] = {};  // start, copied[2], used[2]
    ~CopyPipe() {
        // also where an error ends the streaming: the staging blocks may go to
        // another handle, so no copy into them may be left
        if (cs) cudaStreamSynchronize(cs);
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        if (cs) cudaStreamDestroy(cs);
    }
};
template <typename F>
static void stream_rows(Exec &ex, const double *host, size_t row, int v, F consume) {
    size_t rows_per = (size_t)((512ull << 20) / (row * sizeof(double)));
    if (rows_per < 1) rows_per = 1;
    if (rows_per > (size_t)v) rows_per = v;
    const int nbuf = rows_per < (size_t)v ? 2 : 1;
    double *stage[2] = {nullptr, nullptr};
    for (int b = 0; b < nbuf; b++) dalloc(ex, stage[b], rows_per * row * sizeof(double));
    CopyPipe cp;
    CK(cudaStreamCreateWithFlags(&cp.cs, cudaStreamNonBlocking));
    for (cudaEvent_t &e : cp.ev) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    CK(cudaEventRecord(cp.ev[0], ex.stream));  // the buffers exist in ex.stream's order
    CK(cudaStreamWaitEvent(cp.cs, cp.ev[0], 0));
    int k = 0;
    for (int d0 = 0; d0 < v; d0 += (int)rows_per, k++) {
        const int nr = (int)((size_t)(v - d0) < rows_per ? (size_t)(v - d0) : rows_per);
        const int b = k % nbuf;
        if (k >= nbuf) CK(cudaStreamWaitEvent(cp.cs, cp.ev[3 + b], 0));  // chunk k - nbuf consumed
        CK(cudaMemcpyAsync(stage[b], host + (size_t)d0 * row, nr * row * sizeof(double), cudaMemcpyHostToDevice,
                           cp.cs));
        CK(cudaEventRecord(cp.ev[1 + b], cp.cs));
        CK(cudaStreamWaitEvent(ex.stream, cp.ev[1 + b], 0));
        consume(stage[b], d0, nr);
        CK(cudaEventRecord(cp.ev[3 + b], ex.stream));
    }
    for (int b = 0; b < nbuf; b++) free_tmp(ex, stage[b]);  // synchronises ex.stream
    CK(cudaStreamSynchronize(cp.cs));
}

// The four operand layouts of a problem (tcorr_internal.cuh) in the given element
// kind; vvvo on the host is streamed in chunks of d rows.  pG .. pN: slice plane
// sizes, eA, eB: scale exponents of the two operand sides (FP64 emulation).
static void layout_g(Exec &ex, Problem &pb, int kind, int64_t pG, const int *eA, const double *vvvo, bool host) {
    const int o = pb.dm.o, v = pb.dm.v, dp = pb.dm.dp;
    const int64_t v2 = (int64_t)v * v;
    const size_t eb = kind == 0 ? 8 : (kind == 1 ? 4 : 2);
    Operands &op = pb.op;
    const size_t row = (size_t)v2 * o;  // doubles per d row of vvvo
    // G[q][xy][d] = vvvo[d][xy][q]: rows d, columns (xy, q); the last rows write the padding
    auto g_rows = [&](const double *src, int d0, int nr) {
        char *hi = static_cast<char *>(op.G) + (size_t)d0 * eb;
        char *lo = op.Glo ? static_cast<char *>(op.Glo) + (size_t)d0 * eb : nullptr;
        CK(launch_transpose_rows(kind, src, hi, lo, pG, eA, false, 1, nr, d0 + nr == v ? dp - d0 : nr, (int64_t)row, 0,
                                 (int64_t)row, 0, o, v2 * dp, dp, ex.stream));
    };
    if (!host) g_rows(vvvo, 0, v);
    else stream_rows(ex, vvvo, row, v, g_rows);
}
static void layout_small(Exec &ex, Problem &pb, int kind, int64_t pK, int64_t pR, int64_t pN, const int *eA,
                         const int *eB, const double *dt2, const double *doo) {
    const int o = pb.dm.o, v = pb.dm.v, dp = pb.dm.dp, lp = pb.dm.lp;
    const int64_t v2 = (int64_t)v * v;
    Operands &op = pb.op;
    // T2K[q][xy][l] = t2[q][l][xy]
    CK(launch_transpose_rows(kind, dt2, op.T2K, op.T2Klo, pK, eA, false, o, o, lp, v2, (int64_t)o * v2, v2, v2 * lp, 1, 0, lp,
                             ex.stream));
    // T2R[spa][d] = t2[spa][d]
    CK(launch_pad_convert_rows(kind, dt2, op.T2R, op.T2Rlo, pR, eB, false, (int64_t)o * o * v, v, dp, ex.stream));
    // AoN[qsa][l] = -ooov[l][qsa]
    CK(launch_transpose_rows(kind, doo, op.AoN, op.AoNlo, pN, eB, true, 1, o, lp, (int64_t)o * o * v, 0,
                             (int64_t)o * o * v, 0, 1, 0, lp, ex.stream));
}

// FP64 emulation: the operands as oz_slices() BF16 slice planes under one
// power-of-two scale per operand side (exponents computed on the device from
// max |vvvo|, |t2|, |ooov|, so nothing here waits for the device).
static void build_operands_oz(Exec &ex, Problem &pb, const double *t2, const double *vvvo, const double *ooov,
                              bool host) {
    const int o = pb.dm.o, v = pb.dm.v, dp = pb.dm.dp, lp = pb.dm.lp;
    const int64_t v2 = (int64_t)v * v;
    const size_t S = (size_t)oz_slices();
    const size_t nG = (size_t)o * v2 * dp, nT2K = (size_t)o * v2 * lp;
    const size_t nT2R = (size_t)o * o * v * dp, nAoN = (size_t)o * o * v * lp;
    Operands &op = pb.op;
    dalloc(ex, op.G, nG * 2 * S);
    dalloc(ex, op.T2K, nT2K * 2 * S);
    dalloc(ex, op.T2R, nT2R * 2 * S);
    dalloc(ex, op.AoN, nAoN * 2 * S);
    dalloc(ex, pb.oz_max, 3 * sizeof(unsigned long long));
    dalloc(ex, pb.oz_e, 2 * sizeof(int));
    Timer tm(ex, KC_PREP);
    CK(cudaMemsetAsync(pb.oz_max, 0, 3 * sizeof(unsigned long long), ex.stream));
    double *tmp_t2 = nullptr, *tmp_oo = nullptr;
    const double *dt2 = device_view(ex, t2, (size_t)o * o * v2, host, tmp_t2);
    const double *doo = device_view(ex, ooov, (size_t)o * o * o * v, host, tmp_oo);
    const size_t row = (size_t)v2 * o;  // doubles per d row of vvvo
    if (!host) {
        CK(launch_maxabs(vvvo, (int64_t)(row * v), pb.oz_max, ex.stream));
    } else {
        double m = 0.0;
        bool finite = true;  // std::max passes a NaN over
        for (size_t k = 0; k < row * v; k++) {
            const double a = std::fabs(vvvo[k]);
            m = std::max(m, a);
            finite &= a <= std::numeric_limits<double>::max();
        }
        CK(launch_seed_max(pb.oz_max, finite ? m : std::numeric_limits<double>::infinity(), ex.stream));
    }
    CK(launch_maxabs(dt2, (int64_t)o * o * v2, pb.oz_max + 1, ex.stream));
    CK(launch_maxabs(doo, (int64_t)o * o * o * v, pb.oz_max + 2, ex.stream));
    CK(launch_oz_exponents(pb.oz_max, pb.oz_e, ex.stream));
    const int *eA = pb.oz_e, *eB = pb.oz_e + 1;
    layout_g(ex, pb, 3, (int64_t)nG, eA, vvvo, host);
    layout_small(ex, pb, 3, (int64_t)nT2K, (int64_t)nT2R, (int64_t)nAoN, eA, eB, dt2, doo);
    tm.stop();
    free_tmp(ex, tmp_t2);
    free_tmp(ex, tmp_oo);
}

void build_operands(Exec &ex, Problem &pb, const double *t2, const double *vvvo, const double *ooov,
                    bool host) {
    if (ex.prec == TCORR_FP64_OZ) {
        build_operands_oz(ex, pb, t2, vvvo, ooov, host);
        return;
    }
    const int o = pb.dm.o, v = pb.dm.v, dp = pb.dm.dp, lp = pb.dm.lp;
    const int64_t v2 = (int64_t)v * v;
    const int pprec = operand_prec(ex.prec, o, v);
    const int kind = elem_kind(pprec);
    const size_t eb = elem_bytes(pprec);
    const bool split = ex.prec != TCORR_FP64;
    const size_t nG = (size_t)o * v2 * dp, nT2K = (size_t)o * v2 * lp;
    const size_t nT2R = (size_t)o * o * v * dp, nAoN = (size_t)o * o * v * lp;
    Operands &op = pb.op;
    dalloc(ex, op.G, nG * eb);
    dalloc(ex, op.T2K, nT2K * eb);
    dalloc(ex, op.T2R, nT2R * eb);
    dalloc(ex, op.AoN, nAoN * eb);
    if (split) {
        dalloc(ex, op.Glo, nG * eb);
        dalloc(ex, op.T2Klo, nT2K * eb);
        dalloc(ex, op.T2Rlo, nT2R * eb);
        dalloc(ex, op.AoNlo, nAoN * eb);
    }
    Timer tm(ex, KC_PREP);
    layout_g(ex, pb, kind, 0, nullptr, vvvo, host);
    double *tmp_t2 = nullptr, *tmp_oo = nullptr;
    const double *dt2 = device_view(ex, t2, (size_t)o * o * v2, host, tmp_t2);
    const double *doo = device_view(ex, ooov, (size_t)o * o * o * v, host, tmp_oo);
    layout_small(ex, pb, kind, 0, 0, 0, nullptr, nullptr, dt2, doo);
    tm.stop();
    free_tmp(ex, tmp_t2);
    free_tmp(ex, tmp_oo);
}

void build_epilogue_inputs(Exec &ex, Problem &pb, const double *eps_occ, const double *eps_vir,
                           const double *t1, const double *ovov, bool host) {
    const int o = pb.dm.o, v = pb.dm.v;
    const size_t nov2 = (size_t)o * v * o * v;
    dalloc(ex, pb.eps_o, o * sizeof(double));
    dalloc(ex, pb.eps_v, v * sizeof(double));
    const cudaMemcpyKind kd = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    CK(cudaMemcpyAsync(pb.eps_o, eps_occ, o * sizeof(double), kd, ex.stream));
    CK(cudaMemcpyAsync(pb.eps_v, eps_vir, v * sizeof(double), kd, ex.stream));
    if (fp64_epilogue(ex.prec)) {
        dalloc(ex, pb.t1, (size_t)o * v * sizeof(double));
        dalloc(ex, pb.ovov, nov2 * sizeof(double));
        CK(cudaMemcpyAsync(pb.t1, t1, (size_t)o * v * sizeof(double), kd, ex.stream));
        CK(cudaMemcpyAsync(pb.ovov, ovov, nov2 * sizeof(double), kd, ex.stream));
        if (ex.prec == TCORR_FP64_OZ) {  // the emulation's epilogue works in float-float
            dalloc(ex, pb.evf, (size_t)v * sizeof(float2));
            CK(launch_epilogue_ff_inputs(static_cast<double *>(pb.t1), static_cast<double *>(pb.ovov), pb.eps_v,
                                         pb.oz_max, pb.evf, o, v, ex.stream));
        }
    } else {
        const size_t vp = epi_vp(v);
        dalloc(ex, pb.t1, (size_t)o * vp * sizeof(float));
        dalloc(ex, pb.ovov, (size_t)o * o * vp * vp * sizeof(float));
        dalloc(ex, pb.evf, vp * sizeof(float2));
        double *tmp1 = nullptr, *tmp2 = nullptr;
        const double *d1 = device_view(ex, t1, (size_t)o * v, host, tmp1);
        const double *d2 = device_view(ex, ovov, nov2, host, tmp2);
        CK(launch_epilogue_f32_inputs(d1, d2, pb.eps_v, static_cast<float *>(pb.t1), static_cast<float *>(pb.ovov),
                                      pb.evf, o, v, (int)vp, ex.stream));
        free_tmp(ex, tmp1);
        free_tmp(ex, tmp2);
    }
}

void build_schedule(Exec &ex, Problem &pb) {
    const int64_t o = pb.dm.o;
    pb.ntask = o * (o + 1) * (o + 2) / 6;
    const int nb = (pb.dm.v + EPI_TE - 1) / EPI_TE;
    pb.norb = nb * (nb + 1) * (nb + 2) / 6;
    dalloc(ex, pb.tasks, (size_t)pb.ntask * 3 * sizeof(int));
    dalloc(ex, pb.task_e, (size_t)pb.ntask * 2 * sizeof(double));
    dalloc(ex, pb.orbits, (size_t)pb.norb * 3 * sizeof(int));
    CK(cudaMemsetAsync(pb.task_e, 0, (size_t)pb.ntask * 2 * sizeof(double), ex.stream));
    CK(launch_build_tables(pb.dm.o, nb, pb.tasks, pb.orbits, ex.stream));
}

// Device bytes of one problem's resident data (operands, epilogue inputs, tables).
size_t problem_bytes(const Dims &d, int prec) {
    prec = operand_prec(prec, d.o, d.v);
    const size_t o = d.o, v = d.v, v2 = v * v;
    const size_t eb = elem_bytes(prec), parts = operand_planes(prec);
    size_t b = parts * eb * (o * v2 * d.dp + o * v2 * d.lp + o * o * v * d.dp + o * o * v * d.lp);
    const size_t ve = fp64_epilogue(prec) ? v : (size_t)epi_vp((int)v);  // FP32 inputs are padded
    b += (o * o * ve * ve + o * ve) * u_elem_bytes(prec) + (o + v) * 8 + ve * 8;
    const size_t nb = (v + EPI_TE - 1) / EPI_TE;
    b += nb * (nb + 1) * (nb + 2) / 6 * 12;
    b += o * (o + 1) * (o + 2) / 6 * 28;
    return b;
}
size_t host_staging_bytes(const Dims &d) {
    const size_t o = d.o, v = d.v;
    return std::max<size_t>(o * o * v * v * 8, (size_t)512 << 20);
}

// Tensor-core tile of a problem shape.  Cost model: every (pair tile, N
// pass) unit costs the same, so take the pb with the fewest tiles; ties go to
// pb = 8 (16-wide c rows), then pb = 4.
int model_pb(int v) {
    int best = 8;
    int64_t best_tiles = -1;
    for (int pb : {8, 4, 16}) {
        const int pc = 128 / pb;
        const int64_t t = (int64_t)((v + pb - 1) / pb) * ((v + pc - 1) / pc);
        if (best_tiles < 0 || t < best_tiles) { best = pb; best_tiles = t; }
    }
    return best;
}

void fill_desc(Exec &ex, Problem &pb, int pbt) {
    InstDesc &d = pb.desc;
    d.dm = pb.dm;
    d.norb = pb.norb;
    d.G = pb.op.G;
    d.T2K = pb.op.T2K;
    d.T2R = pb.op.T2R;
    d.AoN = pb.op.AoN;
    d.eps_o = pb.eps_o;
    d.eps_v = pb.eps_v;
    d.t1 = pb.t1;
    d.ovov = pb.ovov;
    d.evf = pb.evf;
    d.tasks = pb.tasks;
    d.orbits = pb.orbits;
    d.task_e = pb.task_e;
    pb.u_task = 3 * pb.dm.ug;
    if (ex.prec == TCORR_FP64) {
        d.f64 = 1;
        pb.gemm_units = f64_units_per_task(pb.dm, 128);
    } else if (ex.prec == TCORR_FP64_OZ) {
        std::string msg;
        if (oz_fill_desc(d, pb.op, pb.oz_e, msg) != cudaSuccess) throw Fail{TCORR_EUNSUPPORTED, msg};
        pb.gemm_units = oz_units_per_task(d);
    } else {
        std::string msg;
        if (tc_fill_desc(d, operand_prec(ex.prec, pb.dm.o, pb.dm.v), pb.op, pbt, TC_KB, ex.pair, msg) != cudaSuccess)
            throw Fail{TCORR_EUNSUPPORTED, msg};
        if (epi_fill_desc(d, msg) != cudaSuccess) throw Fail{TCORR_EUNSUPPORTED, msg};
        pb.gemm_units = tc_units_per_task(d);
    }
}

// The first task (i <= j <= k, lexicographic) with index n of o orbitals
static void task_at(int o, int64_t n, int &i, int &j, int &k) {
    for (i = 0;; i++) {
        const int64_t m = (int64_t)(o - i) * (o - i + 1) / 2;
        if (n < m) break;
        n -= m;
    }
    for (j = i;; j++) {
        const int64_t m = o - j;
        if (n < m) break;
        n -= m;
    }
    k = j + (int)n;
}

int64_t seg_units(const Problem &pb, Seg &sg, PackTabs &tabs) {
    PackTabs::Of of;
    of.run0 = tabs.runs.size();
    of.ent0 = tabs.ents.size();
    tabs.of.push_back(of);
    const InstDesc &d = pb.desc;
    if (d.f64) {
        sg.f64_tp = f64_tile_pairs(pb.dm, sg.ntb);
        return sg.ntb * f64_units_per_task(pb.dm, sg.f64_tp);
    }
    if (!d.packw) return sg.ntb * pb.gemm_units;
    // counting sort of the groups (s; p, q) of the tasks by (p, q).  Packed, the
    // passes are 256 columns wide instead of v, so an SM takes in fewer A rows per
    // product: with it and the scheduler warp of the pair kernel, o=13, v=131 in
    // TF32X3 took 12.4 ms (15.8 before), o=10, v=70 1.03 ms (1.42) and 24 molecules
    // of v = 20..120 28.0 ms (36.7).
    const int o = pb.dm.o;
    std::vector<int> at((size_t)o * o + 1, 0);
    auto each = [&](auto f) {
        int i, j, k;
        task_at(o, sg.task0, i, j, k);
        for (int tb = 0; tb < sg.ntb; tb++) {
            if (i != k) {
                f(tb, 0, i, j, k);
                f(tb, 1, j, i, k);
                f(tb, 2, k, i, j);
            }
            if (++k == o) {
                if (++j == o) j = ++i;
                k = j;
            }
        }
    };
    each([&](int, int, int, int p, int q) { at[(size_t)p * o + q + 1]++; });
    // Side by side only where that saves passes: a run, where it saves an eighth
    // of its own (else its groups one by one, with one B copy per plane instead
    // of one per 16 columns); the segment, where it saves a quarter over all.
    // In the other order (a tile pair's three groups together) two groups share
    // each A slice, which counts for more with few entries per run or large v:
    // 69 consecutive tasks of o=26, v=237 took 9.5 ms so and 9.9 ms in runs.
    auto passes = [&](int n) { return (int)(((int64_t)n * d.packw + 255) / 256); };
    int64_t npass = 0, nent = 0;
    for (size_t m = 0; m < (size_t)o * o; m++) {
        npass += std::min(at[m + 1], passes(at[m + 1]));
        nent += at[m + 1];
    }
    if (4 * npass > 3 * nent) return sg.ntb * pb.gemm_units;
    const int npair = tc_tile_pairs(d);
    int64_t unit = 0;
    for (size_t m = 0; m < (size_t)o * o; m++) {
        const int n = at[m + 1], np = passes(n);
        at[m + 1] += at[m];
        if (n == 0) continue;
        const bool side = 8 * np <= 7 * n;
        for (int e = 0; e < (side ? 1 : n); e++) {
            tabs.runs.push_back(PackRun{(int)unit, at[m] + e, side ? n : 1, side ? np : 1, (int)(m / o), (int)(m % o)});
            unit += (int64_t)npair * (side ? np : 1);
        }
    }
    tabs.ents.resize(of.ent0 + at[(size_t)o * o]);
    each([&](int tb, int g, int s, int p, int q) {
        tabs.ents[of.ent0 + at[(size_t)p * o + q]++] = PackEnt{tb * 4 + g, s};
    });
    sg.nrun = (int)(tabs.runs.size() - of.run0);
    if (unit > 0x7fffffff) throw Fail{TCORR_EUNSUPPORTED, "too many work units in one wave"};
    return unit;
}

void place_tabs(const PackTabs &tabs, std::vector<Seg> &segs, unsigned char *dst, const unsigned char *dev) {
    const size_t rb = tabs.runs.size() * sizeof(PackRun);
    if (rb) memcpy(dst, tabs.runs.data(), rb);
    if (!tabs.ents.empty()) memcpy(dst + rb, tabs.ents.data(), tabs.ents.size() * sizeof(PackEnt));
    for (size_t n = 0; n < segs.size(); n++) {
        segs[n].runs = reinterpret_cast<const PackRun *>(dev) + tabs.of[n].run0;
        segs[n].ents = reinterpret_cast<const PackEnt *>(dev + rb) + tabs.of[n].ent0;
    }
}

Plan make_plan(const Exec &ex, const std::vector<Problem *> &pbs, const std::vector<Span> &spans) {
    Plan pl;
    WaveRec cur{0, 0, 0, 0, 0, 0};
    int64_t u_used = 0, p_used = 0, t_used = 0;
    auto close = [&]() {
        if (cur.nseg > 0) pl.waves.push_back(cur);
        cur = WaveRec{(int)pl.segs.size(), 0, 0, 0, 0, 0};
        u_used = p_used = t_used = 0;
    };
    for (const Span &sp : spans) {
        const Problem &pb = *pbs[sp.inst];
        int64_t t = sp.first, left = sp.count;
        while (left > 0) {
            const int64_t fit_u = (ex.u_cap - u_used) / pb.u_task;
            const int64_t fit_p = (ex.part_cap - p_used) / ((int64_t)pb.norb * 2);
            const int64_t fit_t = ex.wave_tasks - t_used;
            const int64_t fit_e = ((int64_t)0x7fffffff - cur.n_epi) / pb.norb;
            const int64_t n = std::min({left, fit_u, fit_p, fit_t, fit_e});
            if (n <= 0) {
                if (cur.nseg == 0) throw Fail{TCORR_ENOMEM, "wave scratch smaller than one task"};
                close();
                continue;
            }
            Seg s{};
            s.inst = sp.inst;
            s.ntb = (int)n;
            s.task0 = t;
            s.u_off = u_used;
            s.gemm0 = cur.n_gemm;
            s.epi0 = cur.n_epi;
            s.red0 = cur.n_red;
            s.part_off = p_used;
            cur.nseg++;
            cur.tc_brows = std::max(cur.tc_brows, pb.desc.brows);
            cur.n_gemm += seg_units(pb, s, pl.tabs);
            pl.segs.push_back(s);
            cur.n_epi += n * pb.norb;
            cur.n_red += n;
            u_used += n * pb.u_task;
            p_used += n * (int64_t)pb.norb * 2;
            t_used += n;
            t += n;
            left -= n;
        }
        pl.sums.push_back(SumSpan{pb.task_e, sp.first, sp.count, nullptr});
    }
    close();
    return pl;
}

size_t stage_bytes_max(const Exec &ex, const Problem &pb) {
    const int64_t per_wave = std::max<int64_t>(
        1, std::min({ex.u_cap / pb.u_task, ex.part_cap / ((int64_t)pb.norb * 2), ex.wave_tasks, (int64_t)0x7fffffff / pb.norb}));
    const int64_t nseg = (pb.ntask + per_wave - 1) / per_wave + 1;
    return ((size_t)nseg * sizeof(Seg) + 255) / 256 * 256 + 256 + table_bytes_max(pb.dm, ex.prec, ex.pair);
}

size_t table_bytes_max(const Dims &d, int prec, bool pair) {
    // packing has to save a quarter of the passes (seg_units), so packed columns
    // are at most three quarters of a pass wide; a segment has an entry for each of
    // a task's three groups and at most a run per entry
    const int w = is_split(prec) ? tc_pack_width(d.v, pair) : 0;
    if (w == 0 || 4 * w > 3 * 256) return 0;
    const size_t o = d.o;
    return o * (o + 1) * (o + 2) / 6 * 3 * (sizeof(PackRun) + sizeof(PackEnt));
}

void reserve_stage(Exec &ex, size_t bytes) {
    if (bytes <= ex.stage_cap) return;
    CK(cudaStreamSynchronize(ex.stream));  // the old tables may still be in use
    unsigned char *d = ex.d_stage, *h = ex.h_stage;
    ex.d_stage = ex.h_stage = nullptr;  // nothing left to write to where an allocation fails
    ex.stage_cap = 0;
    dfree(ex, d);
    hfree(ex, h);
    dalloc(ex, ex.d_stage, bytes);
    halloc(ex, ex.h_stage, bytes);
    ex.stage_cap = bytes;
}

// Uploads the plan's tables (one copy from pinned staging); returns the
// device segment and span arrays.
void upload_plan(Exec &ex, Plan &pl, Seg *&d_segs, SumSpan *&d_spans) {
    const size_t seg_b = pl.segs.size() * sizeof(Seg);
    const size_t span_off = (seg_b + 255) / 256 * 256;
    const size_t tab_off = (span_off + pl.sums.size() * sizeof(SumSpan) + 255) / 256 * 256;
    const size_t total = tab_off + pl.tabs.bytes();
    if ((int)pl.sums.size() > ex.sums_cap) throw Fail{TCORR_EINVAL, "more spans than the handle was made for"};
    reserve_stage(ex, total);
    for (size_t n = 0; n < pl.sums.size(); n++) pl.sums[n].out = ex.d_sums + 3 * n;
    place_tabs(pl.tabs, pl.segs, ex.h_stage + tab_off, ex.d_stage + tab_off);
    memcpy(ex.h_stage, pl.segs.data(), seg_b);
    memcpy(ex.h_stage + span_off, pl.sums.data(), pl.sums.size() * sizeof(SumSpan));
    CK(cudaMemcpyAsync(ex.d_stage, ex.h_stage, total, cudaMemcpyHostToDevice, ex.stream));
    d_segs = reinterpret_cast<Seg *>(ex.d_stage);
    d_spans = reinterpret_cast<SumSpan *>(ex.d_stage + span_off);
}

// The launch sequence of a plan on stream st (no host synchronisation).
void launch_plan(Exec &ex, const Plan &pl, const Seg *d_segs, const SumSpan *d_spans, cudaStream_t st) {
    for (const WaveRec &wr : pl.waves) {
        Wave w{};
        w.descs = ex.d_descs;
        w.segs = d_segs + wr.seg0;
        w.nseg = wr.nseg;
        w.n_gemm = wr.n_gemm;
        w.n_epi = wr.n_epi;
        w.n_red = wr.n_red;
        w.U = ex.U;
        w.partials = ex.partials;
        w.err = ex.err;
        w.inject_stall = ex.inject_stall;
        w.tc_brows = wr.tc_brows;
        {
            Timer tm(ex, KC_GEMM);
            if (ex.prec == TCORR_FP64) CK(launch_ugemm_f64(w, st));
            else if (ex.prec == TCORR_FP64_OZ) CK(launch_ugemm_oz(ex.sm_count, w, st));
            else CK(launch_ugemm_tc(ex.prec, ex.sm_count, w, st, ex.pair));
            tm.stop();
        }
        {
            Timer tm(ex, KC_EPI);
            CK(launch_epilogue(ex.prec, ex.sm_count, w, st));
            tm.stop();
        }
        {
            Timer tm(ex, KC_RED);
            CK(launch_task_reduce(w, st));
            tm.stop();
        }
    }
    Timer tm(ex, KC_RED);
    CK(launch_span_sums(d_spans, (int)pl.sums.size(), st));
    tm.stop();
}

void raise_err_flag(Exec &ex) {
    if (*ex.h_err) {
        const int e = *ex.h_err;
        *ex.h_err = 0;
        CK(cudaMemsetAsync(ex.err, 0, sizeof(int), ex.stream));
        if (e & (DERR_TIMEOUT_FULL | DERR_TIMEOUT_EMPTY | DERR_TIMEOUT_TMEM))
            throw Fail{TCORR_ETIMEOUT, "device pipeline wait expired (flags " + std::to_string(e) + ")"};
        throw Fail{TCORR_ECUDA, "device reported bad configuration (flags " + std::to_string(e) + ")"};
    }
}
void check_err_flag(Exec &ex) {
    CK(cudaMemcpyAsync(ex.h_err, ex.err, sizeof(int), cudaMemcpyDeviceToHost, ex.stream));
    CK(cudaStreamSynchronize(ex.stream));
    raise_err_flag(ex);
}

// Copies the error flag and the span sums back in one, waits, resolves timers,
// checks the flag.
constexpr size_t RET_SUMS = 64;  // offset of the span sums in the returned block
void finish_call(Exec &ex, int nspans) {
    CK(cudaMemcpyAsync(ex.h_ret, ex.d_ret, RET_SUMS + (size_t)nspans * 3 * sizeof(double), cudaMemcpyDeviceToHost,
                       ex.stream));
    CK(cudaStreamSynchronize(ex.stream));
    resolve_timers(ex);
    raise_err_flag(ex);
}

// ---- create-time helpers ------------------------------------------------------
tcorr_status check_opts(const tcorr_opts &op, std::string &msg) {
    if (op.test_stall != 0 && op.test_stall != 1) {
        msg = "test_stall must be 0 or 1";
        return TCORR_EINVAL;
    }
    if (op.prec < TCORR_FP64 || op.prec > TCORR_FP64_OZ || op.batch_tasks < 0 ||
        (op.host_inputs != 0 && op.host_inputs != 1) || (op.tune != 0 && op.tune != 1) ||
        (op.eager != 0 && op.eager != 1) || op.wave_mb < 0 || (op.single_sm != 0 && op.single_sm != 1)) {
        msg = "invalid option (precision, batch_tasks, host_inputs, tune, eager, wave_mb or single_sm)";
        return TCORR_EINVAL;
    }
    return TCORR_OK;
}

bool sizes_supported(int o, int v) {
    const int64_t v64 = v, o64 = o;
    return !(v64 * v64 * v64 * o64 > ((int64_t)1 << 40) || o > 4096 || v > 8192);
}

void init_exec(Exec &ex, const tcorr_opts &op, void *stream, bool pooled) {
    ex.stream = static_cast<cudaStream_t>(stream);
    ex.prec = op.prec;
    ex.profile = op.profile;
    ex.inject_stall = op.test_stall;
    ex.pair = op.single_sm == 0;
    int dev = 0;
    CK(cudaGetDevice(&dev));
    ex.device = dev;
    if (pooled) {
        ex.pool = handle_pool(dev);
        ex.pool_max = POOL_MAX;
    }
    CK(cudaDeviceGetAttribute(&ex.sm_count, cudaDevAttrMultiProcessorCount, dev));
    CK(cudaDeviceGetAttribute(&ex.cc_major, cudaDevAttrComputeCapabilityMajor, dev));
    CK(cudaDeviceGetAttribute(&ex.cc_minor, cudaDevAttrComputeCapabilityMinor, dev));
    if (ex.prec != TCORR_FP64 && !tc_supported(ex.cc_major, ex.cc_minor))
        throw Fail{TCORR_EUNSUPPORTED, "mixed precision needs the sm_103 tensor-core path (device is sm_" +
                                           std::to_string(ex.cc_major * 10 + ex.cc_minor) + ")"};
    if (is_split(ex.prec)) {  // kernel attributes, before any capture
        CK(tc_prepare(ex.prec));
        CK(epi_prepare());
    }
    if (ex.prec == TCORR_FP64_OZ) CK(oz_prepare());
}

void build_problem(Exec &ex, Problem &pb, int o, int v, const double *eps_occ, const double *eps_vir,
                   const double *t1, const double *t2, const double *vvvo, const double *ooov,
                   const double *ovov, bool host) {
    pb.dm = make_dims(o, v);
    build_operands(ex, pb, t2, vvvo, ooov, host);
    build_epilogue_inputs(ex, pb, eps_occ, eps_vir, t1, ovov, host);
    build_schedule(ex, pb);
}

void alloc_common(Exec &ex, int nspans) {
    const size_t bytes = RET_SUMS + (size_t)nspans * 3 * sizeof(double);
    dalloc(ex, ex.d_ret, bytes);
    halloc(ex, ex.h_ret, bytes);
    ex.err = reinterpret_cast<int *>(ex.d_ret);
    ex.h_err = reinterpret_cast<int *>(ex.h_ret);
    ex.d_sums = reinterpret_cast<double *>(ex.d_ret + RET_SUMS);
    ex.h_sums = reinterpret_cast<double *>(ex.h_ret + RET_SUMS);
    ex.sums_cap = nspans;
    CK(cudaMemsetAsync(ex.err, 0, sizeof(int), ex.stream));
    *ex.h_err = 0;
}

void upload_descs(Exec &ex, const std::vector<Problem *> &pbs) {
    std::vector<InstDesc> hd(pbs.size());
    for (size_t n = 0; n < pbs.size(); n++) hd[n] = pbs[n]->desc;
    dalloc(ex, ex.d_descs, hd.size() * sizeof(InstDesc));
    copy_in(ex, ex.d_descs, hd.data(), hd.size() * sizeof(InstDesc));
}

// Measured tile choice: times the W contraction of a few tasks of the problem
// for each candidate pb and keeps the fastest.  Results are cached per
// (precision, o, v) for the life of the process.
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int>, int> g_tune_cache;

int tuned_pb(Exec &ex, Problem &pb) {
    const int pprec = operand_prec(ex.prec, pb.dm.o, pb.dm.v);
    const auto key = std::make_tuple(pprec * 2 + (ex.pair ? 1 : 0), pb.dm.o, pb.dm.v);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) return it->second;
    }
    // tasks to time: the scratch's worth, at most 16 (skip i = j = k: the first task)
    const int64_t first = pb.ntask > 1 ? 1 : 0;
    const int64_t n = std::max<int64_t>(1, std::min<int64_t>({pb.ntask - first, 16, ex.u_cap / pb.u_task}));
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    int best = model_pb(pb.dm.v);
    float best_ms = -1.f;
    InstDesc *d_one = nullptr;
    Seg *d_seg = nullptr;
    dalloc(ex, d_one, sizeof(InstDesc));
    dalloc(ex, d_seg, sizeof(Seg));
    unsigned char *d_tab = nullptr;
    const size_t tab_cap = (size_t)n * 3 * (sizeof(PackRun) + sizeof(PackEnt));  // at most a run per group
    dalloc(ex, d_tab, tab_cap);
    Problem cp = pb;
    for (int cand : {8, 4, 16}) {
        InstDesc d = pb.desc;
        std::string msg;
        if (tc_fill_desc(d, pprec, pb.op, cand, TC_KB, ex.pair, msg) != cudaSuccess) continue;
        std::vector<Seg> sv(1);
        Seg &s = sv[0];
        s.ntb = (int)n;
        s.task0 = first;
        cp.desc = d;
        cp.gemm_units = tc_units_per_task(d);
        PackTabs tabs;
        const int64_t units = seg_units(cp, s, tabs);
        std::vector<unsigned char> ht(tabs.bytes() + 1);
        place_tabs(tabs, sv, ht.data(), d_tab);
        copy_in(ex, d_tab, ht.data(), tabs.bytes());
        copy_in(ex, d_one, &d, sizeof(InstDesc));
        copy_in(ex, d_seg, &s, sizeof(Seg));
        Wave w{};
        w.descs = d_one;
        w.segs = d_seg;
        w.nseg = 1;
        w.n_gemm = units;
        w.U = ex.U;
        w.err = ex.err;
        w.tc_brows = d.brows;
        float ms_min = -1.f;
        for (int rep = 0; rep < 3; rep++) {
            CK(cudaEventRecord(e0, ex.stream));
            CK(launch_ugemm_tc(ex.prec, ex.sm_count, w, ex.stream, ex.pair));
            CK(cudaEventRecord(e1, ex.stream));
            CK(cudaEventSynchronize(e1));
            float ms = 0.f;
            CK(cudaEventElapsedTime(&ms, e0, e1));
            if (rep > 0 && (ms_min < 0 || ms < ms_min)) ms_min = ms;
        }
        if (best_ms < 0 || ms_min < best_ms * 0.97f) { best = cand; best_ms = ms_min; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    dfree(ex, d_one);
    dfree(ex, d_seg);
    dfree(ex, d_tab);
    check_err_flag(ex);
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = best;
    return best;
}


}  // namespace rt
}  // namespace tcorr
