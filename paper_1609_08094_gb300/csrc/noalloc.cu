// Allocation-free entry point: one task's FP64 energy share from the
// caller's canonical device arrays, with every intermediate in a fixed
// file-scope device array instead of memory obtained from cudaMalloc.
//
// Who needs it: callers that must not allocate device memory themselves or
// through a library -- applications whose device memory is owned entirely by
// their own pool or budget, and latency-sensitive loops that cannot afford
// cudaMalloc/cudaFree, which synchronise the device.  The price is a fixed
// TCORR_NOALLOC_SCRATCH_BYTES array that every GPU loading libtcorr holds
// until the process exits, and a size limit (v <= TCORR_NOALLOC_MAX_V).
//
// Work: a variant of the FP64 W-contraction kernel that reads t2, vvvo and
// ooov in their canonical layouts (no re-laid-out copies, so nothing to
// allocate) and writes the three group tensors U of the task into the
// scratch array; the existing fused epilogue and task reduction then run on
// pointers into the same array and write E[4], E[5] to the caller's output.
#include <mutex>

#include "tcorr_internal.cuh"

namespace tcorr {
namespace {

constexpr int NA_VMAX = TCORR_NOALLOC_MAX_V;
constexpr int NA_TE = 8;                                   // FP64 epilogue cube edge
constexpr int NA_NB = (NA_VMAX + NA_TE - 1) / NA_TE;
constexpr int NA_NORB = NA_NB * (NA_NB + 1) * (NA_NB + 2) / 6;
constexpr size_t NA_U_BYTES = (size_t)3 * NA_VMAX * NA_VMAX * NA_VMAX * sizeof(double);  // 3 ug <= 3 NA_VMAX^3
constexpr size_t NA_PART_OFF = NA_U_BYTES;
constexpr size_t NA_TASK_OFF = NA_PART_OFF + (size_t)NA_NORB * 2 * sizeof(double);
constexpr size_t NA_ORB_OFF = NA_TASK_OFF + 16;
constexpr size_t NA_SEG_OFF = (NA_ORB_OFF + (size_t)NA_NORB * 3 * sizeof(int) + 63) / 64 * 64;
constexpr size_t NA_DESC_OFF = (NA_SEG_OFF + sizeof(Seg) + alignof(InstDesc) - 1) / alignof(InstDesc) * alignof(InstDesc);
constexpr size_t NA_END = NA_DESC_OFF + sizeof(InstDesc);
static_assert(NA_END <= TCORR_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds the declared size");
static_assert(NA_VMAX % UPAD == 0, "maximum v must be a multiple of the U row padding");

// The scratch: U [3][ug] doubles (each group [v][v][vc]), orbit partials [norb][2] doubles,
// the task (3 ints), the block-orbit table [norb][3] ints, and the work
// description the shared epilogue kernels read (one segment, one instance).
static __device__ __align__(256) unsigned char g_noalloc_scratch[TCORR_NOALLOC_SCRATCH_BYTES];

constexpr int MAX_DEVICES = 64;
std::mutex g_mu;
void *g_ptr[MAX_DEVICES] = {};

// Writes the work description, the task and the block orbits A <= B <= C
// (blocks of NA_TE) into the scratch.
__global__ void noalloc_tables_kernel(const InstDesc d, const Seg sg, InstDesc *d_out, Seg *sg_out, int *task,
                                      int *orb, int nb, int i, int j, int k) {
    static_assert(sizeof(InstDesc) % 4 == 0 && sizeof(Seg) % 4 == 0, "word copy");
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&d);
    uint32_t *dst = reinterpret_cast<uint32_t *>(d_out);
    for (int w = threadIdx.x; w < (int)(sizeof(InstDesc) / 4); w += blockDim.x) dst[w] = src[w];
    if (threadIdx.x == 0) {
        *sg_out = sg;
        task[0] = i;
        task[1] = j;
        task[2] = k;
    }
    // thread per (A, B): the triples with this A and B, after those with a smaller
    // first, then second block
    const int a = threadIdx.x / NA_NB, b = threadIdx.x % NA_NB;
    if (a >= nb || b < a || b >= nb) return;
    int n = 0;
    for (int x = 0; x < a; x++) n += (nb - x) * (nb - x + 1) / 2;
    for (int x = a; x < b; x++) n += nb - x;
    for (int c = b; c < nb; c++, n++) {
        orb[3 * n] = a;
        orb[3 * n + 1] = b;
        orb[3 * n + 2] = c;
    }
}
static_assert(NA_NB * NA_NB <= 128, "a thread per (A, B) of the 128");

// U^{s;p,q}[a][b][c] for the three groups of task (i,j,k), FP64, from the
// canonical arrays (same sums as the layout-based FP64 kernel):
//   sum_d t2[s][p][a][d] (db|cq) + sum_d t2[s][q][a][d] (dc|bp)
//   - sum_l (as|lq) t2[p][l][b][c] - sum_l (as|lp) t2[q][l][c][b],
// with (db|cq) = vvvo[d][b][c][q] and (as|lq) = ooov[l][q][s][a].
// Tiles of 32 pairs: at v = 64 the task has 768 of them, 5 on each SM; of 128 pairs
// there were 192, two on some SMs and one on others (v=61: 323 us, 188 so).
constexpr int CT_P = 32, CT_A = 32, CT_K = 8;
__global__ void __launch_bounds__(256) ugemm_f64_canon_kernel(int o, int v, int vc, int64_t ug,
                                                              const double *__restrict__ t2,
                                                              const double *__restrict__ vvvo,
                                                              const double *__restrict__ ooov, int ti, int tj,
                                                              int tk, double *__restrict__ U) {
    __shared__ double As[CT_K][CT_P + 1];
    __shared__ double Bs[CT_K][CT_A + 1];
    if (ti == tj && tj == tk) return;
    const int tid = threadIdx.x;
    const int64_t v2 = (int64_t)v * v;
    const int64_t p0 = (int64_t)blockIdx.x * CT_P;
    const int a0 = blockIdx.y * CT_A;
    const int g = blockIdx.z;
    int s, pp, q;
    if (g == 0) { s = ti; pp = tj; q = tk; }
    else if (g == 1) { s = tj; pp = ti; q = tk; }
    else { s = tk; pp = ti; q = tj; }
    const int tp = tid & 31, ta = tid >> 5;
    double acc[4] = {};
    const int r = tid / CT_K, kk = tid % CT_K;  // the row and k that this thread loads of each operand
    const int64_t pidx = p0 + r;
    const int64_t b = pidx / v, c = pidx % v;
    const int a = a0 + r;
    const int KV = (v + CT_K - 1) / CT_K, KO = (o + CT_K - 1) / CT_K, nch = 2 * KV + 2 * KO;
    double xa = 0.0, xb = 0.0;
    auto load = [&](int ch) {  // chunk ch of K = [d | d | l | l]
        const int seg = ch < KV ? 0 : (ch < 2 * KV ? 1 : (ch < 2 * KV + KO ? 2 : 3));
        const int kx = (ch - (seg == 0 ? 0 : (seg == 1 ? KV : (seg == 2 ? 2 * KV : 2 * KV + KO)))) * CT_K + kk;
        const bool k_in = kx < (seg < 2 ? v : o);
        xa = xb = 0.0;
        if (k_in && pidx < v2) {
            if (seg == 0) xa = vvvo[((kx * (int64_t)v + b) * v + c) * o + q];
            else if (seg == 1) xa = vvvo[((kx * (int64_t)v + c) * v + b) * o + pp];
            else if (seg == 2) xa = t2[(((int64_t)pp * o + kx) * v + b) * v + c];
            else xa = t2[(((int64_t)q * o + kx) * v + c) * v + b];
        }
        if (k_in && a < v) {
            if (seg == 0) xb = t2[(((int64_t)s * o + pp) * v + a) * v + kx];
            else if (seg == 1) xb = t2[(((int64_t)s * o + q) * v + a) * v + kx];
            else if (seg == 2) xb = -ooov[(((int64_t)kx * o + q) * o + s) * v + a];
            else xb = -ooov[(((int64_t)kx * o + pp) * o + s) * v + a];
        }
    };
    load(0);
    for (int ch = 0; ch < nch; ch++) {
        As[kk][r] = xa;
        Bs[kk][r] = xb;
        __syncthreads();
        if (ch + 1 < nch) load(ch + 1);
        if (a0 + ta * 4 < v) {  // a warp whose four a lie past v issues no FMA
#pragma unroll
            for (int k = 0; k < CT_K; k++) {
                const double av = As[k][tp];
#pragma unroll
                for (int x = 0; x < 4; x++) acc[x] = fma(av, Bs[k][ta * 4 + x], acc[x]);
            }
        }
        __syncthreads();
    }
    double *Ug = U + (int64_t)g * ug;
    const int64_t po = p0 + tp;
#pragma unroll
    for (int x = 0; x < 4; x++) {
        const int ax = a0 + ta * 4 + x;
        if (ax < v && po < v2) Ug[((int64_t)ax * v + po / v) * vc + po % v] = acc[x];
    }
}

}  // namespace
}  // namespace tcorr

using namespace tcorr;

extern "C" tcorr_status tcorr_task_energy_noalloc(int o, int v, const double *eps_occ, const double *eps_vir,
                                                  const double *t1, const double *t2, const double *vvvo,
                                                  const double *ooov, const double *ovov, int i, int j, int k,
                                                  double *e_out, void *stream) {
    if (o < 1 || v < 1 || !eps_occ || !eps_vir || !t1 || !t2 || !vvvo || !ooov || !ovov || !e_out)
        return TCORR_EINVAL;
    if (v > TCORR_NOALLOC_MAX_V || o > 4096) return TCORR_EINVAL;  // beyond the fixed scratch
    if (i < 0 || i > j || j > k || k >= o) return TCORR_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return TCORR_ECUDA;
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_ptr[dev]) {  // once per device, with that device current
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
                cudaGetLastError();
                return TCORR_ECUDA;
            }
            g_ptr[dev] = ptr;
        }
        base = g_ptr[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *sc = static_cast<unsigned char *>(base);
    double *U = reinterpret_cast<double *>(sc);
    double *partials = reinterpret_cast<double *>(sc + NA_PART_OFF);
    int *task = reinterpret_cast<int *>(sc + NA_TASK_OFF);
    int *orbits = reinterpret_cast<int *>(sc + NA_ORB_OFF);
    Seg *seg = reinterpret_cast<Seg *>(sc + NA_SEG_OFF);
    InstDesc *desc = reinterpret_cast<InstDesc *>(sc + NA_DESC_OFF);
    const int nb = (v + NA_TE - 1) / NA_TE;
    InstDesc d{};
    d.dm = make_dims(o, v);
    d.norb = nb * (nb + 1) * (nb + 2) / 6;
    d.eps_o = eps_occ;
    d.eps_v = eps_vir;
    d.t1 = t1;
    d.ovov = ovov;
    d.tasks = task;
    d.orbits = orbits;
    d.task_e = e_out;
    Seg sg{};
    sg.inst = 0;
    sg.ntb = 1;
    noalloc_tables_kernel<<<1, 128, 0, st>>>(d, sg, desc, seg, task, orbits, nb, i, j, k);
    const int64_t v2 = (int64_t)v * v;
    dim3 grid((unsigned)((v2 + CT_P - 1) / CT_P), (unsigned)((v + CT_A - 1) / CT_A), 3);
    ugemm_f64_canon_kernel<<<grid, 256, 0, st>>>(o, v, d.dm.vc, d.dm.ug, t2, vvvo, ooov, i, j, k, U);
    Wave w{};
    w.descs = desc;
    w.segs = seg;
    w.nseg = 1;
    w.n_gemm = 0;
    w.n_epi = d.norb;
    w.n_red = 1;
    w.U = U;
    w.partials = partials;
    if (launch_epilogue(TCORR_FP64, 0, w, st) != cudaSuccess) return TCORR_ECUDA;
    if (launch_task_reduce(w, st) != cudaSuccess) return TCORR_ECUDA;
    return cudaGetLastError() == cudaSuccess ? TCORR_OK : TCORR_ECUDA;
}
