// Reading a lattice's state out and moving checkpoints: absolute FP64
// populations from the stored deviations, and plane copies between the padded
// buffer and a dense array.  A warp takes a piece of one row of one plane:
// 32 x READ_PER_LANE elements, all of a lane's loads in flight together.
//
// FP64 without the FP64 unit.  GB300 runs two FP64 operations per clock and
// SM, so one conversion and one addition per population took 2.5 times as
// long as the memory traffic (4096 x 1024 FP32: 241 us for 654 MB).  The sum
// of a constant and an FP32 deviation is formed in integer arithmetic
// instead: a double's bits, read as an integer, count units in the last place
// within its binade, so while the sum stays in the constant's binade its bits
// are the constant's plus the deviation rounded to those units.  Sums that
// leave it (deviations of the order of the constant, in the core of a hot
// jet) take the FP64 operations.  Same bits either way.  4096 x 1024: FP32
// 241 -> 123 us, FP16 moment-split 300 -> 124 (98 and 89 us at the copy rate).
#pragma once

#include "lbm_aa.cuh"

namespace lbm {

constexpr int READ_PER_LANE = 8;

// element offset of node (0, 0) in each of 13 planes
struct PlaneOffsets {
    int64_t off[13];
};

__host__ __device__ __forceinline__ PlaneOffsets ab_planes(int pitch, int64_t plane)
{
    PlaneOffsets p;
    for (int q = 0; q < 13; ++q)
        p.off[q] = q * plane + pitch + PAD_COLS;
    return p;
}

// the windows that hold the post-collision populations of an AA state (aa_post_cell)
__host__ __device__ __forceinline__ PlaneOffsets aa_planes(int phase, int pitch, int64_t plane)
{
    PlaneOffsets p;
    for (int q = 0; q < 13; ++q)
        p.off[q] = aa_post_cell(phase, q, 0, 0, pitch, plane);
    return p;
}

// a constant c > 0 to which FP32 deviations are added
struct AddTo {
    long long bits;  // of c
    float up;        // 2^52 / 2^exponent(c): deviation to units in c's last place
    bool pow2;       // c a power of two: below it the units are half as large
    bool exact;      // the integer path holds (c normal, its last bit 0: ties round as in FP64)
    __device__ __forceinline__ explicit AddTo(double c)
    {
        bits = __double_as_longlong(c);
        const int e = (int)(bits >> 52);  // biased; c > 0
        pow2 = (bits & 0xfffffffffffffll) == 0;
        exact = c > 0.0 && e > 1023 - 40 && e < 1023 + 40 && (bits & 1) == 0;
        up = exact ? __int_as_float((127 + 52 - (e - 1023)) << 23) : 0.f;
    }
};

// bits of the FP64 sum c + v, or false where it leaves c's binade
__device__ __forceinline__ bool add_bits(const AddTo &k, float v, long long &r)
{
    const bool below = k.pow2 && v < 0.f;
    const float x = v * (below ? 2.f * k.up : k.up);
    const unsigned b = __float_as_uint(x);
    // |x| < 2^30: to the nearest integer; beyond, x is one: its mantissa, shifted
    long long q;
    if (fabsf(x) < 1073741824.f) {
        q = __float2int_rn(x);
    } else {
        const int s = min((int)(b >> 23 & 255u) - 150, 39);
        q = (long long)((b & 0x7fffffu) | 0x800000u) << s;
        q = (int)b < 0 ? -q : q;
    }
    r = k.bits + q;
    return k.exact && ((r >> 52) == (k.bits >> 52) - (below ? 1 : 0) || q == 0) && fabsf(x) < 4.5e15f;
}

// population q of a node in FP64, from its deviation v
template <class C>
__device__ __forceinline__ double absolute(const AddTo &k, int q, C v, double rho0, double T0)
{
    if constexpr (std::is_same<C, float>::value) {
        long long r;
        // (a product w rho0 that rounds is fused into the FP64 sum: rho0 = 1 only)
        if ((q >= 9 || rho0 == 1.0) && add_bits(k, v, r))
            return __longlong_as_double(r);
    }
    if (q < 9)
        return (double)v + w9<double>(q) * rho0;
    return (double)v + 0.25 * T0;
}

template <class S>
__global__ void __launch_bounds__(256) state_out_kernel(const S *buf, double *f, double *g, int nx, int nr, int pitch,
                                                        const __grid_constant__ PlaneOffsets planes, double rho0,
                                                        double T0)
{
    using C = compute_t<S>;
    const int lane = threadIdx.x & 31;
    const unsigned item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const unsigned pieces = (unsigned)(nx + 32 * READ_PER_LANE - 1) / (32 * READ_PER_LANE);
    const unsigned row = item / pieces;
    const int q = (int)(row / (unsigned)nr), j = (int)(row - (unsigned)q * (unsigned)nr);
    if (q >= 13)
        return;
    const int i0 = (int)(item - row * pieces) * 32 * READ_PER_LANE + lane;
    const S *src = buf + planes.off[q] + (int64_t)j * pitch;
    double *dst = (q < 9 ? f + (int64_t)q * nr * nx : g + (int64_t)(q - 9) * nr * nx) + (int64_t)j * nx;
    const AddTo k(q < 9 ? w9<double>(q) * rho0 : 0.25 * T0);
    C v[READ_PER_LANE];
#pragma unroll
    for (int n = 0; n < READ_PER_LANE; ++n)
        if (i0 + 32 * n < nx)
            v[n] = load_as<S, C>(src + i0 + 32 * n);
#pragma unroll
    for (int n = 0; n < READ_PER_LANE; ++n)
        if (i0 + 32 * n < nx)
            dst[i0 + 32 * n] = absolute<C>(k, q, v[n], rho0, T0);
}

// moment-split storage: one node per thread (a node's populations share its moments)
template <class S>
__global__ void __launch_bounds__(256) split_state_out_kernel(const S *buf, double *f, double *g, int nx, int nr,
                                                              int pitch, int64_t plane, double rho0, double T0)
{
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= nx)
        return;
    const StepParams<float> lp = lin_params(rho0, T0);
    const float *M = split_m(buf, plane);
    const int64_t N = (int64_t)nx * nr;
    const AddTo k0(w9<double>(0) * rho0), k1(w9<double>(1) * rho0), k5(w9<double>(5) * rho0), kg(0.25 * T0);
    for (int j = blockIdx.y; j < nr; j += gridDim.y) {
        const int64_t o = (int64_t)(j + 1) * pitch + (i + PAD_COLS), n = (int64_t)j * nx + i;
        const float2 jj = reinterpret_cast<const float2 *>(M)[o];
        const float mx = jj.x, mr = jj.y, mT = M[2 * plane + o];
        float d[13];
#pragma unroll
        for (int q = 0; q < 13; ++q)
            d[q] = load_as<S, float>(buf + (int64_t)q * plane + o);
#pragma unroll
        for (int q = 0; q < 13; ++q) {
            const AddTo &k = q == 0 ? k0 : (q < 5 ? k1 : (q < 9 ? k5 : kg));
            const float v = edge_add<float>(lp, q, mx, mr, mT, d[q]);
            (q < 9 ? f + (int64_t)q * N : g + (int64_t)(q - 9) * N)[n] = absolute<float>(k, q, v, rho0, T0);
        }
    }
}

inline unsigned read_blocks(int rows, int nx)
{
    const int64_t items = (int64_t)rows * ((nx + 32 * READ_PER_LANE - 1) / (32 * READ_PER_LANE));
    return (unsigned)((items + 7) / 8);
}

// ---- fields at the current time: Eq. 2 moments of the streamed populations ---------------
// element offsets of the populations streamed into node (0, 0) (stream_cell)
template <class C>
__host__ __device__ inline PlaneOffsets stream_planes(const StepParams<C> &p)
{
    PlaneOffsets o;
    for (int q = 0; q < 13; ++q)
        o.off[q] = stream_cell(p, q, 0, 0);
    return o;
}

__device__ __forceinline__ void put_field(float *o, float v) { *o = v; }
__device__ __forceinline__ void put_field(float *o, double v) { *o = (float)v; }
__device__ __forceinline__ void put_field(double *o, double v) { *o = v; }
__device__ __forceinline__ void put_field(double *o, float v)
{
    *o = (__float_as_uint(v) << 1) == 0 ? __hiloint2double((int)__float_as_uint(v), 0) : diag_double(v);
}

// A node a lane, all of its loads in flight together; a CTA takes 32 columns by eight rows, so
// that the moments of moment-split storage, which the nodes of three rows read, come from L1.
// Bound by memory in FP32.  4096 x 1024 into FP64 / FP32 fields, us, before (a node a thread in
// row order, its position by 64-bit division, the moments again for each population, past L1) ->
// now, and the bytes at the copy rate: FP32 56 / 50 -> 54 / 44 (53 / 43), FP16 49 / 40 -> 45 / 35
// (36 / 26), FP16 moment-split 102 / 99 -> 62 / 50 (44 / 34).  Two nodes a lane: 54 / 44, 47 / 37
// and 77 / 57.
template <class S, class C, class O>
__global__ void __launch_bounds__(256) fields_kernel(const __grid_constant__ StepParams<C> p,
                                                     const __grid_constant__ PlaneOffsets planes, O *out)
{
    const unsigned pieces = (unsigned)(p.nx + 31) / 32, group = blockIdx.x / pieces;
    const int i = (int)(32 * (blockIdx.x - group * pieces) + (threadIdx.x & 31)), j = (int)(8 * group + (threadIdx.x >> 5));
    if (j >= p.nr)
        return;
    const S *src = static_cast<const S *>(p.src) + (int64_t)j * p.pitch;
    Vec<C, 1> f[9], g[4];
    float2 jj[9];
    float T[4];
    if (i < p.nx) {
        if constexpr (IsSplit<S>::value) {  // the moments of the nodes around
            const float *M = split_m(static_cast<const S *>(p.src), p.plane);
            const int64_t o = cell(p, 0, i, j);
#pragma unroll
            for (int q = 1; q < 9; ++q) {
                const int64_t s = o - ey9(q) * p.pitch - ex9(q);
                jj[q] = __ldg(reinterpret_cast<const float2 *>(M) + s);
                if (q < 5)
                    T[q - 1] = __ldg(M + 2 * p.plane + s);
            }
        }
#pragma unroll
        for (int q = 0; q < 9; ++q)
            f[q].x = load_as<S, C>(src + planes.off[q] + i);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            g[q].x = load_as<S, C>(src + planes.off[9 + q] + i);
    }
    const int64_t N = (int64_t)p.nx * p.nr;
    out += (int64_t)j * p.nx;
    // (a branch between the loads and their use keeps all of them in flight: 48 registers for
    // moment-split storage; without it 34, and 74 / 58 us)
    if (i < p.nx) {
        if constexpr (IsSplit<S>::value) {
#pragma unroll
            for (int q = 1; q < 9; ++q)
                f[q].x = edge_add<C>(p, q, jj[q].x, jj[q].y, 0.f, f[q].x);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                g[q].x = pull_add<C>(p, 9 + q, jj[q + 1].x, jj[q + 1].y, T[q], g[q].x);
        }
        const Mom<Vec<C, 1>> m = moments<Vec<C, 1>>(f, g);
        const C rho = p.rho0 + m.drho.x;
        put_field(out + i, rho);
        put_field(out + N + i, m.jx.x / rho);
        put_field(out + 2 * N + i, m.jr.x / rho);
        put_field(out + 3 * N + i, p.T0 + m.dT.x);
    }
}

// ---- checkpoints ---------------------------------------------------------------------
// Rows of `planes` planes between the padded buffer and a dense [plane][row][n]
// array, in words of type U.  One launch instead of a strided copy per plane
// (4096 x 1024 FP32, 436 MB: 13 copies some 290 us, this 60).
template <class U, bool OUT>
__global__ void __launch_bounds__(256) plane_copy_kernel(U *padded, U *dense, int planes, int n, int nr, int pitch,
                                                         const __grid_constant__ PlaneOffsets offs)
{
    constexpr int PER = 4;
    const int lane = threadIdx.x & 31;
    const unsigned item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const unsigned pieces = (unsigned)(n + 32 * PER - 1) / (32 * PER);
    const unsigned row = item / pieces;
    const int q = (int)(row / (unsigned)nr), j = (int)(row - (unsigned)q * (unsigned)nr);
    if (q >= planes)
        return;
    const int i0 = (int)(item - row * pieces) * 32 * PER + lane;
    U *a = padded + offs.off[q] + (int64_t)j * pitch, *b = dense + (int64_t)row * n;
    const U *src = OUT ? a : b;
    U *dst = OUT ? b : a;
    U v[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k)
        if (i0 + 32 * k < n)
            v[k] = src[i0 + 32 * k];
#pragma unroll
    for (int k = 0; k < PER; ++k)
        if (i0 + 32 * k < n)
            dst[i0 + 32 * k] = v[k];
}

template <class U>
inline cudaError_t plane_copy_as(void *padded, void *dense, int planes, int64_t row_bytes, int nr, int64_t pitch_bytes,
                                 const PlaneOffsets &byte_offs, bool out, cudaStream_t s)
{
    PlaneOffsets o;
    for (int q = 0; q < 13; ++q)
        o.off[q] = byte_offs.off[q] / (int64_t)sizeof(U);
    const int n = (int)(row_bytes / (int64_t)sizeof(U));
    const int64_t items = (int64_t)planes * nr * ((n + 127) / 128);
    const unsigned blocks = (unsigned)((items + 7) / 8);
    U *a = static_cast<U *>(padded), *b = static_cast<U *>(dense);
    const int pitch = (int)(pitch_bytes / (int64_t)sizeof(U));
    if (out)
        plane_copy_kernel<U, true><<<blocks, 256, 0, s>>>(a, b, planes, n, nr, pitch, o);
    else
        plane_copy_kernel<U, false><<<blocks, 256, 0, s>>>(a, b, planes, n, nr, pitch, o);
    return cudaGetLastError();
}

// the widest words that every row's two ends and both arrays are aligned to
inline cudaError_t plane_copy(void *padded, void *dense, int planes, int64_t row_bytes, int nr, int64_t pitch_bytes,
                              const PlaneOffsets &byte_offs, bool out, cudaStream_t s)
{
    uint64_t a = (uint64_t)row_bytes | (uint64_t)pitch_bytes | reinterpret_cast<uint64_t>(padded) |
                 reinterpret_cast<uint64_t>(dense);
    for (int q = 0; q < planes; ++q)
        a |= (uint64_t)byte_offs.off[q];
    if (a % 16 == 0)
        return plane_copy_as<uint4>(padded, dense, planes, row_bytes, nr, pitch_bytes, byte_offs, out, s);
    if (a % 8 == 0)
        return plane_copy_as<uint2>(padded, dense, planes, row_bytes, nr, pitch_bytes, byte_offs, out, s);
    if (a % 4 == 0)
        return plane_copy_as<unsigned>(padded, dense, planes, row_bytes, nr, pitch_bytes, byte_offs, out, s);
    if (a % 2 == 0)
        return plane_copy_as<unsigned short>(padded, dense, planes, row_bytes, nr, pitch_bytes, byte_offs, out, s);
    return plane_copy_as<unsigned char>(padded, dense, planes, row_bytes, nr, pitch_bytes, byte_offs, out, s);
}

}  // namespace lbm
