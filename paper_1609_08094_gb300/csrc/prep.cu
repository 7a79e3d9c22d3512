// Layout preparation (S0): re-lays the caller's canonical FP64 blocks into the
// K-major operand layouts of the W-contraction kernels, zero-padding K, and
// for the mixed precisions splits each value x into hi = round(x) and
// lo = round(x - hi) in TF32 or BF16 (the split-precision scheme that replaces
// the paper's dgemm -> sgemm swap of Sec. 3).
#include <cuda_bf16.h>

#include <algorithm>

#include "tcorr_internal.cuh"

namespace tcorr {
namespace {

__device__ __forceinline__ float tf32_rn(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r & 0xFFFFE000u);  // TF32 keeps 10 mantissa bits
}

// Where the values of one output row go: kind 0: hi as FP64; 1, 2: hi and lo planes
// in TF32 (float) or BF16; 3: OZ_PLANES BF16 slice planes `plane` values apart.
struct RowOut {
    void *hi, *lo;
    int64_t plane;
    const int *e;      // kind 3: the scale exponent, on the device
    int neg;           // every value with its sign flipped
};
constexpr int OZ_PLANES = 5, OZ_BITS = 7;
__device__ __forceinline__ double flip(double x, int neg) {
    return __hiloint2double(__double2hiint(x) ^ (neg << 31), __double2loint(x));
}

// T = x 2^(35 - E) rounded to an integer (half to even) and its digits a_1 .. a_5,
// a_p = round half to even of what the digits before leave, times 2^7 each.  The
// same T as from five steps y *= 2^7, a = rint(y), y -= a on y = x 2^-E (the digits
// differ only where one of those lies within 2^-29 of a tie), on the integer pipe:
// FP64 arithmetic runs at 1/64 of its rate, and 15 operations per value bounded
// the pass (o=40, v=300, all layouts: 77.8 ms, now 11.3).
__device__ __forceinline__ int64_t shift_even(int64_t t, int s) {  // t / 2^s, half to even, 1 <= s <= 62
    return (t + (((int64_t)1 << (s - 1)) - 1) + ((t >> s) & 1)) >> s;
}
__device__ __forceinline__ int64_t oz_fixed(double x, int e) {
    const int64_t bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    const int s = 1075 - 35 + e - ex;
    // zero and values below any digit; s < 1: infinity or NaN (eps_ff_kernel answers)
    if (ex == 0 || s > 60 || s < 1) return 0;
    const int64_t m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
    // |x| = m 2^(ex - 1075) < 2^e: T = m 2^-s, s >= 18
    const int64_t t = shift_even(m, s);
    return bits < 0 ? -t : t;
}

// x = a + b with a the top 24 bits of x and b the other 29, cut to 23 with the last
// one sticky, from the bits of x: the FP64 pipe (1/64 of the FP32 rate) bounded
// this pass when the split was done with FP64 conversions and subtractions (o=50,
// v=450 in BF16: 55 ms).  False (a and b unset) for zero and for exponents where b
// would leave FP32's normal range.
__device__ __forceinline__ bool fp32_parts(double x, float &a, float &b) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7ff) - 1023;
    if (ex < -100 || ex > 126) return false;
    const uint32_t sign = hi & 0x80000000u, rest = lo & 0x1fffffffu;
    a = __uint_as_float(sign | (uint32_t)(ex + 127) << 23 | (hi & 0xfffffu) << 3 | lo >> 29);
    const uint32_t base = sign | (uint32_t)(ex + 104) << 23;  // +-2^(ex - 23)
    b = __uint_as_float(base | rest >> 6 | ((rest & 63u) != 0)) - __uint_as_float(base);
    return true;
}
// x = h + l in TF32: h = x rounded to FP32, then to TF32 (ties away); l = x - h likewise
__device__ __forceinline__ void split_tf32(double x, float &h, float &l) {
    float a, b;
    if (fp32_parts(x, a, b)) {
        h = tf32_rn(a + b);
        l = tf32_rn((a - h) + b);  // a - h is exact
    } else {
        h = tf32_rn(static_cast<float>(x));
        l = tf32_rn(static_cast<float>(x - static_cast<double>(h)));
    }
}
// x = h + l in BF16, each rounded to nearest even
__device__ __forceinline__ void split_bf16(double x, __nv_bfloat16 &h, __nv_bfloat16 &l) {
    float a, b;
    if (fp32_parts(x, a, b)) {
        // the rest as a sticky last bit of a: one rounding, as from FP64
        h = __float2bfloat16_rn(b != 0.f ? __uint_as_float(__float_as_uint(a) | 1u) : a);
        // x - h = s + b rounded to odd in FP32 (t + err exact), then once to BF16
        const float s = a - __bfloat162float(h), t = s + b, err = b - (t - s);
        uint32_t u = __float_as_uint(t);
        if (err != 0.f) u = (((__float_as_uint(err) ^ u) >> 31) ? u - 1 : u) | 1u;
        l = __float2bfloat16_rn(__uint_as_float(u));
    } else {
        h = __double2bfloat16(x);
        l = __double2bfloat16(x - static_cast<double>(__bfloat162float(h)));
    }
}

// One value of an output row, and two neighbouring ones (idx even)
template <int KIND>
__device__ __forceinline__ void store_one(const RowOut &o, int e, int64_t idx, double x) {
    if constexpr (KIND == 0) {
        static_cast<double *>(o.hi)[idx] = x;
    } else if constexpr (KIND == 1) {
        split_tf32(x, static_cast<float *>(o.hi)[idx], static_cast<float *>(o.lo)[idx]);
    } else if constexpr (KIND == 2) {
        split_bf16(x, static_cast<__nv_bfloat16 *>(o.hi)[idx], static_cast<__nv_bfloat16 *>(o.lo)[idx]);
    } else {
        int64_t t = oz_fixed(x, e);
#pragma unroll
        for (int p = 0; p < OZ_PLANES; p++) {
            const int s = OZ_BITS * (OZ_PLANES - 1 - p);
            const int64_t a = s ? shift_even(t, s) : t;
            t -= a << s;
            static_cast<__nv_bfloat16 *>(o.hi)[idx + p * o.plane] = __float2bfloat16_rn(static_cast<float>(static_cast<int>(a)));
        }
    }
}
template <int KIND>
__device__ __forceinline__ void store_pair(const RowOut &o, int e, int64_t idx, double x0, double x1) {
    if constexpr (KIND == 0) {
        *reinterpret_cast<double2 *>(static_cast<double *>(o.hi) + idx) = make_double2(x0, x1);
    } else if constexpr (KIND == 1) {
        float2 h, l;
        split_tf32(x0, h.x, l.x);
        split_tf32(x1, h.y, l.y);
        *reinterpret_cast<float2 *>(static_cast<float *>(o.hi) + idx) = h;
        *reinterpret_cast<float2 *>(static_cast<float *>(o.lo) + idx) = l;
    } else if constexpr (KIND == 2) {
        __nv_bfloat162 h, l;
        split_bf16(x0, h.x, l.x);
        split_bf16(x1, h.y, l.y);
        *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(o.hi) + idx) = h;
        *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(o.lo) + idx) = l;
    } else {
        int64_t t0 = oz_fixed(x0, e), t1 = oz_fixed(x1, e);
        __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(o.hi) + idx;
#pragma unroll
        for (int p = 0; p < OZ_PLANES; p++) {
            const int s = OZ_BITS * (OZ_PLANES - 1 - p);
            const int64_t a0 = s ? shift_even(t0, s) : t0, a1 = s ? shift_even(t1, s) : t1;
            t0 -= a0 << s;
            t1 -= a1 << s;
            __nv_bfloat162 d;
            d.x = __float2bfloat16_rn(static_cast<float>(static_cast<int>(a0)));
            d.y = __float2bfloat16_rn(static_cast<float>(static_cast<int>(a1)));
            *reinterpret_cast<__nv_bfloat162 *>(out + p * o.plane) = d;
        }
    }
}

// Rows r of the input become the innermost index of the output:
//   out[b ob + (c % m) s1 + (c / m) s2 + r] = conv(+-in[b sb + r sr + c]),
// r < R, zero for R <= r < Rp (Rp even, or the last r of a row without padding).
// A CTA takes 32 neighbouring c (256-byte reads) and all r (or, where there are few
// c, some: gridDim.y), 64 at a time through shared memory; each output row gets
// runs of 64 r.  All layouts of o=50, v=450 (45 GB in, 22 GB out in BF16) took 97 ms
// when each (x, y) was a transpose of its own d x q with q in 32-wide tiles, after a
// pass that zeroed the output, and take 23 ms; in FP64 61 and 19 ms.
constexpr int TC = 32, TR = 64;
template <int KIND>
__global__ void __launch_bounds__(256) transpose_rows_kernel(const double *__restrict__ in, const RowOut o, int R, int Rp,
                                                             int64_t C, int64_t sb, int64_t sr, int64_t ob, uint32_t m,
                                                             int64_t s1, int64_t s2, int odd) {
    __shared__ __align__(16) double tile[TC][TR + 2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nct = (C + TC - 1) / TC;
    const int e = KIND == 3 ? o.e[0] : 0;
    const int64_t b = blockIdx.x / nct, c0 = (blockIdx.x - b * nct) * TC;
    const double *src = in + b * sb + c0 + lane;
    const bool c_in = c0 + lane < C;
    for (int r0 = blockIdx.y * TR; r0 < Rp; r0 += gridDim.y * TR) {
        const int nr = min(TR, Rp - r0);
#pragma unroll
        for (int k = 0; k < TR / 8; k++) {
            const int r = r0 + warp + 8 * k;
            if (warp + 8 * k < nr) tile[lane][warp + 8 * k] = c_in && r < R ? flip(src[(int64_t)r * sr], o.neg) : 0.0;
        }
        __syncthreads();
        // lanes along r, two values each: 8, 16 or 32 lanes per output row
        const int sh = nr <= 16 ? 3 : (nr <= 32 ? 4 : 5);
        const int r = 2 * (threadIdx.x & ((1 << sh) - 1));
        for (int cc = threadIdx.x >> sh; cc < TC; cc += 256 >> sh) {
            const int64_t c = c0 + cc;
            if (c >= C || r >= nr) continue;
            const int64_t row = b * ob + (m == 1 ? c * s2 : (int64_t)((uint32_t)c % m) * s1 + (int64_t)((uint32_t)c / m) * s2) + r0;
            if (!odd && r + 1 < nr) {
                store_pair<KIND>(o, e, row + r, tile[cc][r], tile[cc][r + 1]);
            } else {  // rows that start on odd values, or the last of an odd number
                store_one<KIND>(o, e, row + r, tile[cc][r]);
                if (r + 1 < nr) store_one<KIND>(o, e, row + r + 1, tile[cc][r + 1]);
            }
        }
        __syncthreads();
    }
}

// out[row Rp + r] = conv(+-in[row R + r]), zero for R <= r < Rp (Rp even): a warp per row
template <int KIND>
__global__ void __launch_bounds__(256) pad_convert_rows_kernel(const double *__restrict__ in, const RowOut o,
                                                               int64_t rows, int R, int Rp) {
    const int lane = threadIdx.x & 31;
    const int e = KIND == 3 ? o.e[0] : 0;
    for (int64_t row = blockIdx.x * 8 + (threadIdx.x >> 5); row < rows; row += (int64_t)gridDim.x * 8) {
        const double *src = in + row * R;
        for (int r = 2 * lane; r < Rp; r += 64)
            store_pair<KIND>(o, e, row * Rp + r, r < R ? flip(src[r], o.neg) : 0.0, r + 1 < R ? flip(src[r + 1], o.neg) : 0.0);
    }
}

// FP32 epilogue inputs of the split-precision paths, the virtual extents
// padded with zeros to vp (a multiple of the epilogue's cube edge 8): (p x | q z)
// as [p][q][X][Z][8][8], so that each of an orbit's 8x8 sub-blocks is one
// contiguous, aligned 256-byte bulk copy, and t1 as rows [p][x].
__global__ void ovov_blocks_kernel(const double *__restrict__ in, float *__restrict__ out, int o, int v,
                                   int vp) {
    const int64_t n = (int64_t)o * o * vp * vp;
    const int nb = vp / 8;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int lz = (int)(i & 7), lx = (int)((i >> 3) & 7);
        int64_t r = i >> 6;
        const int zb = (int)(r % nb);
        r /= nb;
        const int xb = (int)(r % nb);
        r /= nb;
        const int q = (int)(r % o), pp = (int)(r / o);
        const int x = xb * 8 + lx, z = zb * 8 + lz;
        out[i] = (x < v && z < v) ? static_cast<float>(in[(((int64_t)pp * v + x) * o + q) * v + z]) : 0.f;
    }
}

// eps_v as float-float pairs: hi = eps rounded to FP32, lo = the rest rounded
// to FP32 (about 48 significant bits together); zero for x >= v
// eps_v as float-float pairs.  m (FP64 emulation, else NULL): the bits of the largest
// |vvvo|, |t2| and |ooov|.  A digit plane has no infinity or NaN, so such a value
// would leave finite energies behind: eps_v[0], which every task's denominators
// read, becomes NaN then, and with it every energy of the problem.
__global__ void eps_ff_kernel(const double *__restrict__ e, const unsigned long long *__restrict__ m,
                              float2 *__restrict__ out, int v, int vp) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= vp) return;
    double d = x < v ? e[x] : 0.0;
    if (m && x == 0) {
        const unsigned long long inf = 0x7ff0000000000000ull;
        if (m[0] >= inf || m[1] >= inf || m[2] >= inf) d = __longlong_as_double(0x7ff8000000000000ll);
    }
    const float hi = static_cast<float>(d);
    out[x] = make_float2(hi, static_cast<float>(d - static_cast<double>(hi)));
}

// FP64 values to float-float pairs in place (the same 8 bytes per value)
__global__ void to_ff_kernel(double *__restrict__ x, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double d = x[i];
        const float hi = static_cast<float>(d);
        reinterpret_cast<float2 *>(x)[i] = make_float2(hi, static_cast<float>(d - static_cast<double>(hi)));
    }
}

__global__ void pad_rows_kernel(const double *__restrict__ in, float *__restrict__ out, int rows, int v,
                                int vp) {
    const int64_t n = (int64_t)rows * vp;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % vp);
        out[i] = x < v ? static_cast<float>(in[(i / vp) * v + x]) : 0.f;
    }
}

}  // namespace

cudaError_t launch_transpose_rows(int kind, const double *in, void *out_hi, void *out_lo, int64_t plane, const int *e,
                                  bool negate, int64_t B, int R, int Rp, int64_t C, int64_t sb, int64_t sr, int64_t ob,
                                  int64_t m, int64_t s1, int64_t s2, cudaStream_t st) {
    const int64_t grid = B * ((C + TC - 1) / TC);
    if (grid == 0 || Rp == 0) return cudaSuccess;
    if (grid > 0x7fffffff || (m > 1 && C > 0xffffffffll)) return cudaErrorInvalidValue;
    const RowOut o{out_hi, out_lo, plane, e, negate ? 1 : 0};
    // pairs are stored as one: every row has to start on an even value of a plane
    const size_t pair = kind == 0 ? 16 : (kind == 1 ? 8 : 4);
    const int odd = ((uintptr_t)out_hi | (uintptr_t)out_lo) % pair != 0 || ob % 2 != 0 || (m > 1 && s1 % 2 != 0) ||
                    s2 % 2 != 0 || plane % 2 != 0;
    const int ny = (int)std::min<int64_t>((Rp + TR - 1) / TR, std::max<int64_t>(1, 1024 / grid));
    const dim3 gd((unsigned)grid, (unsigned)ny);
#define TR_LAUNCH(K) transpose_rows_kernel<K><<<gd, 256, 0, st>>>(in, o, R, Rp, C, sb, sr, ob, (uint32_t)m, s1, s2, odd)
    if (kind == 0) TR_LAUNCH(0);
    else if (kind == 1) TR_LAUNCH(1);
    else if (kind == 2) TR_LAUNCH(2);
    else TR_LAUNCH(3);
#undef TR_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_pad_convert_rows(int kind, const double *in, void *out_hi, void *out_lo, int64_t plane, const int *e,
                                    bool negate, int64_t rows, int R, int Rp, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    if (Rp % 2 != 0 || plane % 2 != 0) return cudaErrorInvalidValue;
    const RowOut o{out_hi, out_lo, plane, e, negate ? 1 : 0};
    const unsigned grid = (unsigned)(rows / 8 < 8192 ? (rows + 7) / 8 : 8192);
    if (kind == 0) pad_convert_rows_kernel<0><<<grid, 256, 0, st>>>(in, o, rows, R, Rp);
    else if (kind == 1) pad_convert_rows_kernel<1><<<grid, 256, 0, st>>>(in, o, rows, R, Rp);
    else if (kind == 2) pad_convert_rows_kernel<2><<<grid, 256, 0, st>>>(in, o, rows, R, Rp);
    else pad_convert_rows_kernel<3><<<grid, 256, 0, st>>>(in, o, rows, R, Rp);
    return cudaGetLastError();
}

cudaError_t launch_epilogue_ff_inputs(double *t1, double *ovov, const double *eps_v, const unsigned long long *m,
                                      float2 *evf, int o, int v, cudaStream_t st) {
    const int64_t n = (int64_t)o * v * o * v, blocks = (n + 255) / 256;
    to_ff_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(ovov, n);
    to_ff_kernel<<<(unsigned)(((int64_t)o * v + 255) / 256), 256, 0, st>>>(t1, (int64_t)o * v);
    eps_ff_kernel<<<(v + 255) / 256, 256, 0, st>>>(eps_v, m, evf, v, v);
    return cudaGetLastError();
}

cudaError_t launch_epilogue_f32_inputs(const double *t1, const double *ovov, const double *eps_v, float *t1f,
                                       float *ovf, float2 *evf, int o, int v, int vp, cudaStream_t st) {
    if (vp % 8 != 0 || vp < v) return cudaErrorInvalidValue;
    const int64_t n = (int64_t)o * o * vp * vp, blocks = (n + 255) / 256;
    ovov_blocks_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(ovov, ovf, o, v, vp);
    pad_rows_kernel<<<(unsigned)((o * (int64_t)vp + 255) / 256), 256, 0, st>>>(t1, t1f, o, v, vp);
    eps_ff_kernel<<<(vp + 255) / 256, 256, 0, st>>>(eps_v, nullptr, evf, v, vp);
    return cudaGetLastError();
}


namespace {
// Thread per (x, y): the sorted triples x <= y <= z of n values with this x and
// y, in lexicographic order after the T(n) - T(n - x) triples with a smaller first
// index, T(m) = m (m + 1) (m + 2) / 6, and those with this x and a smaller second.
__global__ void sorted_triples_kernel(int n, int *out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int x = (int)(t / n), y = (int)(t % n);
    if (x >= n || y < x) return;
    const int64_t m = n - x, k = n - y, N = n;
    int64_t off = N * (N + 1) * (N + 2) / 6 - m * (m + 1) * (m + 2) / 6 + m * (m + 1) / 2 - k * (k + 1) / 2;
    int *w = out + 3 * off;
    for (int z = y; z < n; z++) {
        w[0] = x;
        w[1] = y;
        w[2] = z;
        w += 3;
    }
}
}  // namespace

cudaError_t launch_build_tables(int o, int nb, int *tasks, int *orbits, cudaStream_t st) {
    sorted_triples_kernel<<<(unsigned)(((int64_t)o * o + 63) / 64), 64, 0, st>>>(o, tasks);
    sorted_triples_kernel<<<(unsigned)(((int64_t)nb * nb + 63) / 64), 64, 0, st>>>(nb, orbits);
    return cudaGetLastError();
}

}  // namespace tcorr
