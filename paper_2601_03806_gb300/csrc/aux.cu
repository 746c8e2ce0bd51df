// aux.cu -- non-hot kernels: initial state, AA-aware gather/scatter of the
// populations, moment export (Eqs. rho/u and Pi), observable fields and the
// shell binning of S(k) (Sec. III; sums as good as FP64's, FP64 totals), and
// the final pass of the fused reductions.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "error_free.cuh"
#include "internal.h"
#include "stats.cuh"
#include "lattice.cuh"
#include "step_kernel.cuh"

namespace flbm {

namespace {

__device__ __forceinline__ void node_xyz(uint64_t n, const BoxDesc &b, uint32_t &x, uint32_t &y,
                                         uint32_t &z)
{
    if (b.n <= 0xffffffffull) {   // 32-bit divisions
        const uint32_t m = uint32_t(n), r = m / b.nx;
        x = m - r * b.nx;
        z = r / b.ny;
        y = r - z * b.ny;
        return;
    }
    x = uint32_t(n % b.nx);
    const uint64_t r = n / b.nx;
    y = uint32_t(r % b.ny);
    z = uint32_t(r / b.ny);
}

__device__ __forceinline__ uint32_t wrap(uint32_t v, int d, uint32_t L)
{
    if (d > 0) return (v + 1 < L) ? v + 1 : 0;
    if (d < 0) return v ? v - 1 : L - 1;
    return v;
}

// Storage index of f_i(x, t) for the current parity: natural form keeps it in
// slot i at x; the AA odd form keeps it in slot opp(i) at x - c_i.
__device__ __forceinline__ uint64_t storage_index(int cx, int cy, int cz, uint32_t x, uint32_t y,
                                                  uint32_t z, const BoxDesc &b)
{
    if (b.parity == 0) {
        const uint64_t n = x + uint64_t(b.nx) * (y + uint64_t(b.ny) * z);
        return uint64_t(slot_of(cx, cy, cz)) * b.ns + n;
    }
    const uint32_t xx = wrap(x, -cx, b.nx), yy = wrap(y, -cy, b.ny), zz = wrap(z, -cz, b.nz);
    const uint64_t n = xx + uint64_t(b.nx) * (yy + uint64_t(b.ny) * zz);
    return uint64_t(slot_of(-cx, -cy, -cz)) * b.ns + n;
}

// storage element <-> double
template <typename S>
__device__ __forceinline__ double to_d(S v) { return double(v); }
template <>
__device__ __forceinline__ double to_d<__half>(__half v) { return double(__half2float(v)); }
template <typename S>
__device__ __forceinline__ S from_d(double v) { return S(v); }
template <>
__device__ __forceinline__ __half from_d<__half>(double v) { return __float2half_rn(float(v)); }

template <typename S>
__device__ __forceinline__ double ldd(const S *g, uint64_t i) { return to_d(g[i]); }

// Arithmetic type of the auxiliary kernels: double for FP64 storage, float
// otherwise (the deviations are O(1e-2) and the storage is FP32 / FP16
// anyway; FP64 arithmetic is the slow pipe on this GPU).
template <typename S>
using Acc = typename std::conditional<std::is_same<S, double>::value, double, float>::type;

template <typename S>
__device__ __forceinline__ Acc<S> lda(const S *g, uint64_t i) { return Acc<S>(to_d(g[i])); }
template <>
__device__ __forceinline__ float lda<float>(const float *g, uint64_t i) { return g[i]; }
template <>
__device__ __forceinline__ float lda<__half>(const __half *g, uint64_t i) { return __half2float(g[i]); }



template <typename S>
__global__ void k_fill_zero(S *g, uint64_t count)
{
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < count;
         i += uint64_t(gridDim.x) * blockDim.x)
        g[i] = from_d<S>(0.0);
}

// out[i*cn + k] = f_i (absolute, or deviation) at node n0 + k
template <typename S>
__global__ void k_gather_f(const S *g, BoxDesc b, uint64_t n0, uint64_t cn, double *out)
{
    for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < cn;
         k += uint64_t(gridDim.x) * blockDim.x) {
        uint32_t x, y, z;
        node_xyz(n0 + k, b, x, y, z);
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz) {
                    const int i = slot_of(cx, cy, cz);
                    const double w = w1(cx) * w1(cy) * w1(cz);
                    const double gv = ldd(g, storage_index(cx, cy, cz, x, y, z, b));
                    out[uint64_t(i) * cn + k] = gv + w * b.rho0;
                }
    }
}

template <typename S>
__global__ void k_gather_state(const S *g, BoxDesc b, uint64_t n0, uint64_t cn, S *out)
{
    for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < cn;
         k += uint64_t(gridDim.x) * blockDim.x) {
        uint32_t x, y, z;
        node_xyz(n0 + k, b, x, y, z);
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz)
                    out[uint64_t(slot_of(cx, cy, cz)) * cn + k] =
                        g[storage_index(cx, cy, cz, x, y, z, b)];
    }
}

// natural-form write of f_i - w_i rho0 from in[i*cn + k]
template <typename S>
__global__ void k_scatter_f(S *g, BoxDesc b, uint64_t n0, uint64_t cn, const double *in)
{
    for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < cn;
         k += uint64_t(gridDim.x) * blockDim.x) {
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz) {
                    const int i = slot_of(cx, cy, cz);
                    const double w = w1(cx) * w1(cy) * w1(cz);
                    g[uint64_t(i) * b.ns + n0 + k] = from_d<S>(in[uint64_t(i) * cn + k] - w * b.rho0);
                }
    }
}

// Natural-form thermal sample g_i = sqrt(rho0 kT w_i / c_s^2) xi_i.
template <typename S>
__global__ void k_init_thermal(S *g, BoxDesc b, double kT, uint32_t key0, uint32_t key1)
{
    uint32_t rk[20];
    for (int r = 0; r < 10; ++r) {
        rk[2 * r] = key0 + uint32_t(r) * 0x9E3779B9u;
        rk[2 * r + 1] = key1 + uint32_t(r) * 0xBB67AE85u;
    }
    using A = Acc<S>;
    const A base = A(sqrt(b.rho0 * kT * 3.0));   // sqrt(rho0 kT / c_s^2)
    for (uint64_t n = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; n < b.n;
         n += uint64_t(gridDim.x) * blockDim.x) {
        A xi[28];
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            const u32x4 o = philox4x32_10(u32x4{uint32_t(n), 0u, uint32_t(6 + j), 0u}, rk);
            A rad, c, sn;
            box_muller(o.x, o.y, rad, c, sn);
            xi[4 * j] = rad * c;
            xi[4 * j + 1] = rad * sn;
            box_muller(o.z, o.w, rad, c, sn);
            xi[4 * j + 2] = rad * c;
            xi[4 * j + 3] = rad * sn;
        }
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz) {
                    const int i = slot_of(cx, cy, cz);
                    // sqrt(w_i) = prod sqrt(w1): sqrt(2/3), sqrt(1/6)
                    const double sw = (cx ? 0.40824829046386302 : 0.81649658092772603) *
                                      (cy ? 0.40824829046386302 : 0.81649658092772603) *
                                      (cz ? 0.40824829046386302 : 0.81649658092772603);
                    g[uint64_t(i) * b.ns + n] = from_d<S>(double(base * A(sw) * xi[i]));
                }
    }
}

// out[k*27 + i] = f_i (absolute) at node nodes[k]
template <typename S>
__global__ void k_probe(const S *g, BoxDesc b, const long long *nodes, long long count, double *out)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
         k += (long long)gridDim.x * blockDim.x) {
        uint32_t x, y, z;
        node_xyz(uint64_t(nodes[k]), b, x, y, z);
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz) {
                    const int i = slot_of(cx, cy, cz);
                    const double w = w1(cx) * w1(cy) * w1(cz);
                    out[k * 27 + i] = ldd(g, storage_index(cx, cy, cz, x, y, z, b)) + w * b.rho0;
                }
    }
}

// Pre-collision moments: out planes rho, jx, jy, jz, Pxx, Pyy, Pzz, Pxy, Pxz,
// Pyz (FP64; Pi = sum f c c includes the rest part rho0 c_s^2 delta).
template <typename S>
__global__ void k_moments(const S *g, BoxDesc b, uint64_t n0, uint64_t cn, double *out)
{
    using A = Acc<S>;
    for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < cn;
         k += uint64_t(gridDim.x) * blockDim.x) {
        uint32_t x, y, z;
        node_xyz(n0 + k, b, x, y, z);
        A m[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx)
#pragma unroll
            for (int cy = -1; cy <= 1; ++cy)
#pragma unroll
                for (int cz = -1; cz <= 1; ++cz) {
                    const A gv = lda(g, storage_index(cx, cy, cz, x, y, z, b));
                    m[0] += gv;
                    if (cx) m[1] += cx * gv;
                    if (cy) m[2] += cy * gv;
                    if (cz) m[3] += cz * gv;
                    if (cx) m[4] += gv;
                    if (cy) m[5] += gv;
                    if (cz) m[6] += gv;
                    if (cx && cy) m[7] += (cx * cy) * gv;
                    if (cx && cz) m[8] += (cx * cz) * gv;
                    if (cy && cz) m[9] += (cy * cz) * gv;
                }
        const double pr = b.rho0 / 3.0;   // rest-state c_s^2 rho0 on the diagonal
        out[0 * cn + k] = b.rho0 + double(m[0]);
        out[1 * cn + k] = double(m[1]);
        out[2 * cn + k] = double(m[2]);
        out[3 * cn + k] = double(m[3]);
        out[4 * cn + k] = pr + double(m[4]);
        out[5 * cn + k] = pr + double(m[5]);
        out[6 * cn + k] = pr + double(m[6]);
        out[7 * cn + k] = double(m[7]);
        out[8 * cn + k] = double(m[8]);
        out[9 * cn + k] = double(m[9]);
    }
}

// Weight of velocity (cx, cy, cz) in observable OBS (flbm_observable).
template <int OBS>
__device__ __forceinline__ constexpr int obs_weight(int cx, int cy, int cz)
{
    return OBS == 0   ? 1
           : OBS == 1 ? cx + cy + cz
           : OBS == 2 ? cx * cx + cy * cy + cz * cz
           : OBS == 3 ? cx * cy + cx * cz + cy * cz
           : OBS == 4 ? cx
           : OBS == 5 ? cy
                      : cz;
}
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// V consecutive storage elements (one 16-byte load for V > 1) as Acc<S>.
template <typename S, int V>
__device__ __forceinline__ void load_vec(const S *p, Acc<S> (&v)[V])
{
    if constexpr (V == 1) {
        v[0] = lda(p, 0);
    } else {
        const uint4 raw = __ldg(reinterpret_cast<const uint4 *>(p));
        S e[V];
        memcpy(e, &raw, sizeof(raw));
#pragma unroll
        for (int q = 0; q < V; ++q) v[q] = lda(e, q);
    }
}

// Observable field m(x) (deviation from the rest state; the constant offset
// only affects the excluded n = 0 mode) and the largest |m|, as the bits of a
// float, into *peak.  HBM-bound: it reads the 18 to 27 slabs its weights
// touch.  The observable is a template argument, so every load of a node is
// issued before the first is used; as a run-time switch inside the loop each
// waited for the one before (256^3: 854 us, a quarter of the copy rate).  Nine
// loads at a time in 64 registers: four CTAs per SM keep more of them in
// flight than all 27 at once do (256^3, four observables: 1.58 ms, 1.74).  In
// the natural form nodes are taken V at a time (one 16-byte load per slab,
// V = 16 / element size); the AA-shifted form shifts them along x, so one at
// a time (V = 1).
template <typename S, typename F, int OBS, int V>
__global__ void __launch_bounds__(256, 4) k_observable(const S *__restrict__ g, const BoxDesc b, F *__restrict__ field,
                                                    unsigned int *peak)
{
    using A = Acc<S>;
    float top = 0.0f;
    const uint64_t groups = b.n / V;
    for (uint64_t q = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; q < groups;
         q += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t n = q * V;
        uint32_t x = 0, y = 0, z = 0;
        if (V == 1) node_xyz(n, b, x, y, z);
        A acc[V];
#pragma unroll
        for (int e = 0; e < V; ++e) acc[e] = 0;
#pragma unroll
        for (int cx = -1; cx <= 1; ++cx) {
            A v[9][V];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const int cy = q / 3 - 1, cz = q % 3 - 1;
                if (obs_weight<OBS>(cx, cy, cz) != 0)
                    load_vec<S, V>(g + (V == 1 ? storage_index(cx, cy, cz, x, y, z, b)
                                               : uint64_t(slot_of(cx, cy, cz)) * b.ns + n),
                                   v[q]);
            }
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const int c = obs_weight<OBS>(cx, q / 3 - 1, q % 3 - 1);
                if (c != 0)
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[e] = fma_(A(c), v[q][e], acc[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < V; ++e) {
            field[n + e] = F(acc[e]);
            top = fmaxf(top, fabsf(float(acc[e])));
        }
    }
    // non-negative floats compare as their bits
    const unsigned int bits = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
    if ((threadIdx.x & 31) == 0 && bits) atomicMax(peak, bits);
}

// ---------------------------------------------------------------------------
// Shell binning of the R2C spectrum [nz][ny][nx/2+1] (complex of T).

__device__ __forceinline__ ShellSum<float> shell_up(const ShellSum<float> &v, int d)
{
    return ShellSum<float>{__shfl_up_sync(0xffffffffu, v.hi, d), __shfl_up_sync(0xffffffffu, v.mid, d),
                           __shfl_up_sync(0xffffffffu, v.lo, d)};
}
__device__ __forceinline__ ShellSum<double> shell_up(const ShellSum<double> &v, int d)
{
    return ShellSum<double>{__shfl_up_sync(0xffffffffu, v.v, d)};
}

// k of the power of two 2^k that brings a spectrum whose field peaks at `peak`
// (its bits) into a range where FP32 squares neither overflow nor underflow:
// every amplitude is at most N peak, and so is the root of the sum of all
// squares (Parseval); N peak goes to about 2^60.  Exact, and divided out of
// the totals.
__device__ __forceinline__ int shell_scale(unsigned int peak, uint64_t n)
{
    if (peak == 0u || peak >= 0x7f800000u) return 0;
    const int k = 60 - (int(peak >> 23) - 127 + 1) - (64 - __clzll((long long)n));
    return k > 126 ? 126 : (k < -126 ? -126 : k);
}
__device__ __forceinline__ float power2(int k, float) { return __uint_as_float(uint32_t(127 + k) << 23); }
__device__ __forceinline__ double power2(int k, double) { return __longlong_as_double((long long)(1023 + k) << 52); }

// round(|n|) of n2 = |n|^2: 0, or the s >= 1 with s^2 - s < n2 <= s^2 + s (|n|
// is never a half-integer), from a square root good to one.
__device__ __forceinline__ long long shell_of(unsigned long long n2)
{
    if (n2 == 0) return 0;
    long long s = n2 < (1ull << 44) ? (long long)(__fsqrt_rn(float(n2)) + 0.5f) : llrint(sqrt(double(n2)));
    while (s * s - s >= (long long)n2) --s;
    while (s * s + s < (long long)n2) ++s;
    return s;
}

// The same for n2 < 2^31, in 32 bits.
__device__ __forceinline__ uint32_t shell_of(uint32_t n2)
{
    if (n2 == 0) return 0;
    uint32_t s = uint32_t(__fsqrt_rn(float(n2)) + 0.5f);
    while (s * s - s >= n2) --s;
    while (s * s + s < n2) ++s;
    return s;
}

constexpr int kShellWarps = 8;
constexpr size_t kShellSmem = 200 * 1024;
// Bytes of a bin (a sum and a count), and warps of a CTA whose private bins fit.
template <typename T>
constexpr size_t kShellBin = sizeof(ShellSum<T>) + sizeof(unsigned int);
template <typename T>
int shell_warps(int nshell)
{
    const size_t w = kShellSmem / (size_t(nshell) * kShellBin<T>);
    return w < size_t(kShellWarps) ? int(w) : kShellWarps;
}

// The lane's sum of the squares of up to four complex elements.
__device__ __forceinline__ ShellSum<float> square_sum(const float (&re)[4], const float (&im)[4])
{
    TripleSum<float2> w;   // real and imaginary parts, a lane each
    w.hi = w.mid = w.lo = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < 4; ++q) w.add_square(make_float2(re[q], im[q]));
    ShellSum<float> v;
    v.hi = w.hi.x;
    v.mid = w.mid.x;
    v.lo = w.lo.x + w.lo.y;
    v.add(w.hi.y, w.mid.y);
    return v;
}
__device__ __forceinline__ ShellSum<double> square_sum(const double (&re)[4], const double (&im)[4])
{
    ShellSum<double> v;
    v.zero();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v.add_square(re[q]);
        v.add_square(im[q]);
    }
    return v;
}

// A warp takes the rows kx = 0 .. nx/2 of (+-ky, +-kz), up to four at once:
// they have the same |n| element by element, so one shell index and one
// binning serve four values.  Along a row the shell only grows, so lanes of
// one shell are neighbours: a segmented scan, as deep as the longest segment
// needs, leaves each shell's sum on its last lane, which adds it to the warp's
// own bins in shared memory -- no atomics until the CTA's totals, added in
// FP64.  Rows stop at the last shell asked for.  Bound by instruction issue:
// 256^3, 129 shells, 30 us (FP32) and 39 us (FP64); element by element in FP64
// (k_shells_flat) 322 and 300 us.
template <typename T>
__global__ void __launch_bounds__(32 * kShellWarps) k_shells(const T *__restrict__ spec, const BoxDesc b, int nshell,
                                                             double inv_n, const unsigned int *peak, double *S,
                                                             unsigned long long *cnt)
{
    extern __shared__ __align__(16) unsigned char shell_raw[];
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ShellSum<T> *const sums = reinterpret_cast<ShellSum<T> *>(shell_raw);
    unsigned int *const cnts = reinterpret_cast<unsigned int *>(shell_raw + size_t(warps) * nshell * sizeof(ShellSum<T>));
    for (int i = threadIdx.x; i < warps * nshell; i += blockDim.x) {
        sums[i].zero();
        cnts[i] = 0u;
    }
    __syncthreads();
    using C = typename std::conditional<std::is_same<T, float>::value, float2, double2>::type;
    const C *const elems = reinterpret_cast<const C *>(spec);
    ShellSum<T> *const bin = sums + size_t(warp) * nshell;
    unsigned int *const num = cnts + size_t(warp) * nshell;
    const uint32_t nxh = b.nx / 2 + 1, nyh = b.ny / 2 + 1, nzh = b.nz / 2 + 1;
    auto square = [](uint64_t v) { return v * v; };
    // every |n|^2, of the lanes past a row's end too, is below 2^31
    const bool narrow = square(nxh + 31) + square(nyh) + square(nzh) < (uint64_t(1) << 31);
    const int k2 = std::is_same<T, float>::value ? shell_scale(*peak, b.n) : 0;
    const T scale = power2(k2, T(0));
    // rows r = warp's index, + warps in all, ...: (ay, az) = (r % nyh, r / nyh), stepped without a division
    const uint32_t first = blockIdx.x * uint32_t(warps) + warp, step = gridDim.x * uint32_t(warps);
    uint32_t ay = first % nyh, az = first / nyh;
    auto next = [&] {
        ay += step % nyh;
        az += step / nyh;
        if (ay >= nyh) {
            ay -= nyh;
            ++az;
        }
    };
    for (; az < nzh; next()) {
        const bool two_y = ay != 0 && 2 * uint64_t(ay) != b.ny, two_z = az != 0 && 2 * uint64_t(az) != b.nz;
        const unsigned long long perp = (unsigned long long)ay * ay + (unsigned long long)az * az;
        const int mult = (two_y ? 2 : 1) * (two_z ? 2 : 1);
        const C *row[4];   // (ky, kz), (-ky, kz), (ky, -kz), (-ky, -kz)
        row[0] = elems + (uint64_t(az) * b.ny + ay) * nxh;
        row[1] = elems + (uint64_t(az) * b.ny + (b.ny - ay)) * nxh;
        row[2] = elems + (uint64_t(b.nz - az) * b.ny + ay) * nxh;
        row[3] = elems + (uint64_t(b.nz - az) * b.ny + (b.ny - ay)) * nxh;
        for (uint32_t k0 = 0; k0 < nxh; k0 += 32) {
            const uint32_t kx = k0 + lane;
            const long long s = narrow ? (long long)shell_of(kx * kx + uint32_t(perp))
                                       : shell_of((unsigned long long)kx * kx + perp);
            const bool in = kx < nxh && s < nshell;
            // lanes of one row: in holds on a prefix of the warp
            const unsigned int on = __ballot_sync(0xffffffffu, in);
            if (!on) break;
            // the conjugate half (kx -> -kx) has the same |n|; kx = 0 and the
            // even Nyquist plane are their own partners
            const bool own = kx == 0 || (b.nx % 2 == 0 && kx == b.nx / 2);
            T re[4], im[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool use = in && (!(q & 1) || two_y) && (!(q & 2) || two_z);
                const C f = use ? row[q][kx] : C{};
                re[q] = f.x * scale;
                im[q] = f.y * scale;
            }
            ShellSum<T> v = square_sum(re, im);
            if (!own) v.scale2();
            const int sh = in ? int(s) : -1;
            const int left = __shfl_up_sync(0xffffffffu, sh, 1);
            const unsigned int heads = __ballot_sync(0xffffffffu, in && (lane == 0 || left != sh));
            const unsigned int owns = __ballot_sync(0xffffffffu, in && own);
            const unsigned int upto = 0xffffffffu >> (31 - lane);        // lanes 0 .. lane
            const int head = in ? 31 - __clz(int(heads & upto)) : lane;
            // bit l of runs: lanes l - d .. l are of one shell
            unsigned int runs = on & ~heads;
            for (int d = 1; runs; d <<= 1) {
                const ShellSum<T> o = shell_up(v, d);
                if (lane - d >= head) v.add(o);
                runs &= runs << d;
            }
            const bool tail = in && (lane == 31 || (((heads | ~on) >> (lane + 1)) & 1u));
            if (tail && sh > 0) {   // shell 0 holds only n = 0, which is excluded
                const unsigned int seg = upto & ~((1u << head) - 1u);
                bin[sh].add(v);
                num[sh] += unsigned(mult) * (2u * __popc(seg) - __popc(owns & seg));
            }
            __syncwarp();
        }
    }
    __syncthreads();
    const double inv = inv_n * power2(-2 * k2, 0.0);
    for (int s = threadIdx.x; s < nshell; s += blockDim.x) {
        double t = 0.0;
        unsigned long long k = 0;
        for (int w = 0; w < warps; ++w) {
            const unsigned int c = cnts[size_t(w) * nshell + s];
            if (!c) continue;   // most, where a warp takes a row or two
            t += sums[size_t(w) * nshell + s].value();
            k += c;
        }
        if (k) {
            atomicAdd(&S[s], t * inv);
            atomicAdd(&cnt[s], k);
        }
    }
}

// The same sums element by element, in FP64, into the CTA's bins in shared
// memory by atomics: for spectra whose rows are too few, or too short, to fill
// the warps of k_shells (shells_flat).
template <typename T>
__global__ void __launch_bounds__(256) k_shells_flat(const T *__restrict__ spec, const BoxDesc b, int nshell,
                                                     double inv_n, double *S, unsigned long long *cnt)
{
    extern __shared__ __align__(16) unsigned char shell_raw[];
    double *const sums = reinterpret_cast<double *>(shell_raw);
    unsigned long long *const cnts = reinterpret_cast<unsigned long long *>(sums + nshell);
    for (int s = threadIdx.x; s < nshell; s += blockDim.x) {
        sums[s] = 0.0;
        cnts[s] = 0ull;
    }
    __syncthreads();
    const uint32_t nxh = b.nx / 2 + 1;
    const uint64_t total = uint64_t(nxh) * b.ny * b.nz;
    for (uint64_t e = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; e < total;
         e += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t kx = uint32_t(e % nxh);
        const uint64_t r = e / nxh;
        const uint32_t ky = uint32_t(r % b.ny), kz = uint32_t(r / b.ny);
        const unsigned long long ay = min(ky, b.ny - ky), az = min(kz, b.nz - kz);
        const long long s = shell_of((unsigned long long)kx * kx + ay * ay + az * az);
        if (s == 0 || s >= nshell) continue;
        const double re = double(spec[2 * e]), im = double(spec[2 * e + 1]);
        const unsigned int wgt = (kx == 0 || (b.nx % 2 == 0 && kx == b.nx / 2)) ? 1u : 2u;
        atomicAdd(&sums[s], wgt * (re * re + im * im) * inv_n);
        atomicAdd(&cnts[s], (unsigned long long)wgt);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nshell; s += blockDim.x) {
        if (cnts[s]) {
            atomicAdd(&S[s], sums[s]);
            atomicAdd(&cnt[s], cnts[s]);
        }
    }
}

// Whether the shells are summed element by element: where a row has one or two
// elements (1 x 1024 x 1024, 513 shells: 35 us, 187 by rows; 1 x 1 x 2^20, 3072
// shells: 16 and 431; with three, 4 x 512 x 512, 257 shells, FP32: 49 and 40),
// and where rows are long and the elements few.  A warp takes about a
// microsecond for 32 elements of a row, in which k_shells_flat adds 29,000, and
// rows go side by side: 4096 x 16 x 16, 2049 shells: 19 us, 109 by rows; 1000 x
// 30 x 20, 501 shells: 14 and 33; 1024 x 1024 x 1, 513 shells, just beyond the
// line: 29 and 30.  Below four chunks the rows win whatever their number (8^3:
// 9 us and 5).
inline bool shells_flat(const BoxDesc &b, int nshell)
{
    const uint64_t nxh = b.nx / 2 + 1, chunks = std::min<uint64_t>((nxh + 31) / 32, uint64_t(nshell) / 32 + 1);
    return nxh <= 2 || (chunks >= 4 && nxh * b.ny * b.nz < 29000 * chunks);
}

// Training pairs: for every node the features x_i = g_i / sqrt(rho0 kT w_i /
// c_s^2), x_27 = omega - 1, and the targets
//   t_i = w_i sum_{k >= 10} e_ki rho u^(deg k) / b_k / (w_i sigma^3),
// the ghost equilibrium content by which the regularized collision (Reg-FLBM)
// differs from the GMF collision of the same pre-collision state, in FP64.
//
// The FP64 pipe bounds it (two operations per clock and SM), so the kernel is
// arranged around its count, about 270 a node instead of 1044: the density
// and momentum come from axis-wise partial sums (49 additions, not 81); the
// 17 ghost amplitudes are products of per-axis factors kappa_a u^a; the
// synthesis skips the modes below order 3; 1 / w_i, a power of four times a
// constant, goes into the amplitudes and, exactly, into the FP32 results;
// and 1 / sqrt(w_i) into four host constants.  A CTA's rows of X and T are
// contiguous, so they leave through shared memory in whole lines.
struct PairConst {
    double x[4];        // 1 / sqrt(rho0 kT w / c_s^2) for |c|^2 = 0, 1, 2, 3
    double scale;       // 27/8 / sigma^3: 1 / w_i = 27/8 4^(|c|^2)
    float x27;          // omega - 1
};

// 1-D synthesis (step_kernel.cuh) of a line whose degree-0 (and, with Z1,
// degree-1) amplitude is zero.
template <bool Z1>
__device__ __forceinline__ void synthesise_high(double &p0, double &p1, double &p2)
{
    const double t = p2, z = -2.0 * p2;
    p0 = Z1 ? t : t - p1;
    p2 = Z1 ? t : t + p1;
    p1 = z;
}

constexpr int kPairBlock = 128;

template <typename S>
__global__ void __launch_bounds__(kPairBlock) k_mlp_pairs(const S *__restrict__ g, const BoxDesc b, const PairConst c,
                                                          float *__restrict__ X, float *__restrict__ T)
{
    __shared__ float row[kPairBlock * 28];
    for (uint64_t n0 = uint64_t(blockIdx.x) * kPairBlock; n0 < b.n; n0 += uint64_t(gridDim.x) * kPairBlock) {
        const uint64_t n = n0 + threadIdx.x;
        const uint32_t live = uint32_t(b.n - n0 < kPairBlock ? b.n - n0 : kPairBlock);
        const bool on = threadIdx.x < live;
        double d[3][3][3];
        uint32_t x, y, z;
        node_xyz(on ? n : n0, b, x, y, z);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    d[i][j][k] = ldd(g, storage_index(i - 1, j - 1, k - 1, x, y, z, b));
                    row[threadIdx.x * 28 + slot_of(i - 1, j - 1, k - 1)] =
                        float(d[i][j][k] * c.x[(i != 1) + (j != 1) + (k != 1)]);
                }
        row[threadIdx.x * 28 + 27] = c.x27;
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < live * 28; e += kPairBlock) X[n0 * 28 + e] = row[e];
        // rho and j from sums along x, then y, then z
        double sx[3][3], dx[3], s[3], jx = 0.0, jy = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double m[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                sx[j][k] = (d[0][j][k] + d[2][j][k]) + d[1][j][k];
                m[j] = d[2][j][k] - d[0][j][k];
            }
            dx[k] = (m[0] + m[2]) + m[1];
            s[k] = (sx[0][k] + sx[2][k]) + sx[1][k];
            jy += sx[2][k] - sx[0][k];
        }
        jx = (dx[0] + dx[2]) + dx[1];
        const double rho = b.rho0 + ((s[0] + s[2]) + s[1]);
        const double jz = s[2] - s[0];
        const double ir = 1.0 / rho;
        // per-axis factors kappa_a u^a (kappa = 2/3, 1/2, 1/2), rho and the
        // scale in the x axis's
        const double u[3] = {jx * ir, jy * ir, jz * ir}, r = rho * c.scale;
        double f[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double pre = a == 0 ? r : 1.0;
            f[a][0] = kappa1d(0) * pre;
            f[a][1] = (kappa1d(1) * pre) * u[a];
            f[a][2] = f[a][1] * u[a];
        }
        double q[3][3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const double fij = f[0][i] * f[1][j];
#pragma unroll
                for (int k = 0; k < 3; ++k) q[i][j][k] = mode_order(i, j, k) >= 3 ? fij * f[2][k] : 0.0;
            }
        // z, y and x passes; lines and entries below order 3 are zero
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if (i + j == 1) synthesise_high<true>(q[i][j][0], q[i][j][1], q[i][j][2]);
                else if (i + j == 2) synthesise_high<false>(q[i][j][0], q[i][j][1], q[i][j][2]);
                else if (i + j > 2) synthesise(q[i][j][0], q[i][j][1], q[i][j][2]);
            }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            synthesise_high<false>(q[0][0][k], q[0][1][k], q[0][2][k]);
            synthesise(q[1][0][k], q[1][1][k], q[1][2][k]);
            synthesise(q[2][0][k], q[2][1][k], q[2][2][k]);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) synthesise(q[0][j][k], q[1][j][k], q[2][j][k]);
        __syncthreads();   // X has left the staging rows
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int far = (i != 1) + (j != 1) + (k != 1);
                    row[threadIdx.x * 27 + slot_of(i - 1, j - 1, k - 1)] =
                        float(q[i][j][k]) * (far == 0 ? 1.0f : far == 1 ? 4.0f : far == 2 ? 16.0f : 64.0f);
                }
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < live * 27; e += kPairBlock) T[n0 * 27 + e] = row[e];
        __syncthreads();   // T has left before the next nodes' X
    }
}

// Totals of the fused reductions of up to kStatSlots steps: CTA (s, i) adds
// sum s of slot i's per-CTA partials in a fixed order, and the CTA that
// finishes last (no CTA waits) adds the steps to the accumulators in step
// order, a thread per component.  One launch per kStatSlots steps, and 13
// CTAs per step because FP64 adds run at two per clock and SM: one CTA per
// step took 15-17 us a step, a seventh of the 128^3 step and most of the 64^3
// one; with the means' divisions in parallel this takes under 1 us a step.
__global__ void __launch_bounds__(kStatThreads) k_stats_finalize(const StatBatch f, DevStats *st, double n)
{
    __shared__ double red[kStatSlots * kStatTerms];   // at least kStatThreads
    static_assert(kStatSlots * kStatTerms >= kStatThreads, "the sums use it too");
    __shared__ double tot[kStatSlots * NSTAT];
    __shared__ bool last;
    const int s = blockIdx.x, i = blockIdx.y, t = threadIdx.x;
    const double sum = stat_total(f.partials + size_t(i) * f.slot_stride + s, f.nblocks[i], red);
    if (t == 0) {
        f.totals[i * NSTAT + s] = sum;
        __threadfence();
        last = atomicAdd(f.arrived, 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int e = t; e < int(gridDim.y) * NSTAT; e += kStatThreads) tot[e] = __ldcg(f.totals + e);   // other SMs' too
    __syncthreads();
    stats_update(st, tot, int(gridDim.y), f.step, n, red);
    if (t == 0) *f.arrived = 0u;
}

inline int grid_for(uint64_t work, int block)
{
    uint64_t g = (work + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 65535ull * 16) g = 65535ull * 16;
    return int(g);
}

}  // namespace

// Calls f with a value of the storage type of precision code prec
// (0 double, 1 float, 2 half).
template <typename F>
void with_storage(int prec, F &&f)
{
    if (prec == 0) f(double{});
    else if (prec == 1) f(float{});
    else f(__half{});
}

cudaError_t launch_fill_rest(void *g, int prec, uint64_t count, cudaStream_t s)
{
    const int grid = grid_for(count, 256) > 4096 ? 4096 : grid_for(count, 256);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_fill_zero<S><<<grid, 256, 0, s>>>(static_cast<S *>(g), count);
    });
    return cudaGetLastError();
}

cudaError_t launch_gather_f(const void *g, int prec, const BoxDesc &b, uint64_t n0, uint64_t cn,
                            double *out, cudaStream_t s)
{
    const int grid = grid_for(cn, 128);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_gather_f<S><<<grid, 128, 0, s>>>(static_cast<const S *>(g), b, n0, cn, out);
    });
    return cudaGetLastError();
}

cudaError_t launch_gather_state(const void *g, int prec, const BoxDesc &b, uint64_t n0, uint64_t cn,
                                void *out, cudaStream_t s)
{
    const int grid = grid_for(cn, 128);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_gather_state<S><<<grid, 128, 0, s>>>(static_cast<const S *>(g), b, n0, cn, static_cast<S *>(out));
    });
    return cudaGetLastError();
}

cudaError_t launch_scatter_f(void *g, int prec, const BoxDesc &b, uint64_t n0, uint64_t cn,
                             const double *in, cudaStream_t s)
{
    const int grid = grid_for(cn, 128);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_scatter_f<S><<<grid, 128, 0, s>>>(static_cast<S *>(g), b, n0, cn, in);
    });
    return cudaGetLastError();
}

cudaError_t launch_mlp_pairs(const void *g, int prec, const BoxDesc &b, double kT, double omega, float *X, float *T,
                             cudaStream_t s)
{
    const int grid = grid_for(b.n, kPairBlock);
    const double w[4] = {8.0 / 27.0, 2.0 / 27.0, 1.0 / 54.0, 1.0 / 216.0}, sig = std::sqrt(kT / b.rho0);
    PairConst c;
    for (int k = 0; k < 4; ++k) c.x[k] = 1.0 / std::sqrt(b.rho0 * kT * w[k] * 3.0);
    c.scale = 3.375 / (sig * sig * sig);
    c.x27 = float(omega - 1.0);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_mlp_pairs<S><<<grid, kPairBlock, 0, s>>>(static_cast<const S *>(g), b, c, X, T);
    });
    return cudaGetLastError();
}

cudaError_t launch_init_thermal(void *g, int prec, const BoxDesc &b, double kT, uint64_t seed,
                                cudaStream_t s)
{
    const int grid = grid_for(b.n, 128) > 8192 ? 8192 : grid_for(b.n, 128);
    const uint32_t k0 = uint32_t(seed & 0xffffffffu), k1 = uint32_t(seed >> 32);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_init_thermal<S><<<grid, 128, 0, s>>>(static_cast<S *>(g), b, kT, k0, k1);
    });
    return cudaGetLastError();
}

cudaError_t launch_probe(const void *g, int prec, const BoxDesc &b, const long long *nodes,
                         long long count, double *out, cudaStream_t s)
{
    const int grid = grid_for(uint64_t(count), 128);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_probe<S><<<grid, 128, 0, s>>>(static_cast<const S *>(g), b, nodes, count, out);
    });
    return cudaGetLastError();
}

cudaError_t launch_moments(const void *g, int prec, const BoxDesc &b, uint64_t n0, uint64_t cn,
                           double *out, cudaStream_t s)
{
    const int grid = grid_for(cn, 128);
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        k_moments<S><<<grid, 128, 0, s>>>(static_cast<const S *>(g), b, n0, cn, out);
    });
    return cudaGetLastError();
}

namespace {
template <typename S, int V>
void observable(const void *g, const BoxDesc &b, int obs, void *field, unsigned int *peak, int grid, cudaStream_t s)
{
    using F = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    const S *p = static_cast<const S *>(g);
    F *f = static_cast<F *>(field);
    switch (obs) {
    case 0: k_observable<S, F, 0, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    case 1: k_observable<S, F, 1, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    case 2: k_observable<S, F, 2, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    case 3: k_observable<S, F, 3, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    case 4: k_observable<S, F, 4, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    case 5: k_observable<S, F, 5, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    default: k_observable<S, F, 6, V><<<grid, 256, 0, s>>>(p, b, f, peak); break;
    }
}
}  // namespace

// The observable field is double for FP64 storage and float otherwise.
cudaError_t launch_observable(const void *g, int prec, const BoxDesc &b, int obs, void *field, unsigned int *peak,
                              cudaStream_t s)
{
    with_storage(prec, [&](auto tag) {
        using S = decltype(tag);
        constexpr int V = 16 / int(sizeof(S));
        // 16-byte loads: natural form, whole groups of V, every slab (256-byte
        // aligned buffer) starting on 16 bytes
        const bool vec = b.parity == 0 && b.n % V == 0 && b.ns % V == 0;
        const uint64_t groups = vec ? b.n / V : b.n;
        const int grid = int(std::min<uint64_t>((groups + 255) / 256, uint64_t(b.nsm) * 16));
        if (vec) observable<S, V>(g, b, obs, field, peak, grid, s);
        else observable<S, 1>(g, b, obs, field, peak, grid, s);
    });
    return cudaGetLastError();
}

cudaError_t launch_shells(const void *spec, int prec, const BoxDesc &b, int nshell, const unsigned int *peak, double *S,
                          unsigned long long *cnt, cudaStream_t s)
{
    const double inv_n = 1.0 / double(b.n);   // a division costs the kernels a microsecond
    auto run = [&](auto zero) {
        using T = decltype(zero);
        if (shells_flat(b, nshell)) {
            const uint64_t total = uint64_t(b.nx / 2 + 1) * b.ny * b.nz;
            const int grid = int(std::min<uint64_t>((total + 255) / 256, 2048));
            k_shells_flat<T><<<grid, 256, size_t(nshell) * (sizeof(double) + sizeof(unsigned long long)), s>>>(
                static_cast<const T *>(spec), b, nshell, inv_n, S, cnt);
            return;
        }
        const int warps = shell_warps<T>(nshell);
        const uint64_t rows = uint64_t(b.ny / 2 + 1) * (b.nz / 2 + 1);
        const int grid = int(std::min<uint64_t>((rows + warps - 1) / warps, uint64_t(b.nsm) * 4));
        cudaFuncSetAttribute(k_shells<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kShellSmem));
        k_shells<T><<<grid, 32 * warps, warps * nshell * kShellBin<T>, s>>>(static_cast<const T *>(spec), b, nshell,
                                                                            inv_n, peak, S, cnt);
    };
    if (prec == 0) run(0.0);
    else run(0.0f);
    return cudaGetLastError();
}

cudaError_t launch_stats_finalize(const StatBatch &f, int slots, DevStats *st, double n, cudaStream_t s)
{
    k_stats_finalize<<<dim3(NSTAT, unsigned(slots)), kStatThreads, 0, s>>>(f, st, n);
    return cudaGetLastError();
}

}  // namespace flbm
