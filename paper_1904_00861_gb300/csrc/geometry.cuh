// Pair geometry shared by the kernels that walk neighbour lists: separations
// in FP64 (minimum image) and from FP32 cell offsets, the cell shift of a list
// entry, the kernel gradient and F_ij of a pair, and the packed neighbour
// records.
#pragma once

#include "pair_terms.cuh"

namespace dtsph {

// r_ij in FP64 with the minimum image; returns |r_ij|^2 (no FMA contraction).
template <int D>
__device__ __forceinline__ double sep64(const Geom &G, const double *x, int n, int i, int j, double *d)
{
#pragma unroll
    for (int a = 0; a < D; ++a) {
        double v = __dsub_rn(x[(size_t)a * n + i], x[(size_t)a * n + j]);
        if (G.periodic[a]) {
            if (v > G.halfL[a]) v = __dsub_rn(v, G.L[a]);
            else if (v < -G.halfL[a]) v = __dadd_rn(v, G.L[a]);
        }
        d[a] = v;
    }
    double r2 = __dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1]));
    if (D == 3) r2 = __dadd_rn(r2, __dmul_rn(d[2], d[2]));
    return r2;
}

// FP32 separation from cell offsets: the own offset is first moved by the cell
// shift (dx, dy, dz) s, then the neighbour's offset is subtracted; both the
// traversal test and the pair terms use this form, so they see the same bits.
template <int D>
__device__ __forceinline__ float4 shifted_offset(float4 oi, int dx, int dy, int dz, const float *sf)
{
    using A = Ar<float>;
    float4 p;
    p.x = A::fma(-(float)dx, sf[0], oi.x);
    p.y = A::fma(-(float)dy, sf[1], oi.y);
    p.z = D == 3 ? A::fma(-(float)dz, sf[2], oi.z) : 0.f;
    p.w = 0.f;
    return p;
}

template <int D>
__device__ __forceinline__ float sep32(float4 ps, float4 oj, float &f0, float &f1, float &f2)
{
    using A = Ar<float>;
    f0 = A::sub(ps.x, oj.x);
    f1 = A::sub(ps.y, oj.y);
    f2 = D == 3 ? A::sub(ps.z, oj.z) : 0.f;
    float q2 = A::fma(f1, f1, A::mul(f0, f0));
    if (D == 3) q2 = A::fma(f2, f2, q2);
    return q2;
}

// r_ij and |r_ij|^2 in the working precision T of a listed neighbour j (cell
// shift (dx, dy, dz)), with the arithmetic of the traversal test.
template <int D, bool F32, typename T>
__device__ __forceinline__ void listed_sep(const Geom &G, const double *__restrict__ x, const float4 *__restrict__ off,
                                           int n, int i, int j, float4 oi, int dx, int dy, int dz, T *d, T &r2)
{
    if (F32) {
        float f0, f1, f2;
        const float q2 = sep32<D>(shifted_offset<D>(oi, dx, dy, dz, G.s_f), off[j], f0, f1, f2);
        d[0] = (T)f0;
        d[1] = (T)f1;
        if (D == 3) d[2] = (T)f2;
        r2 = (T)q2;
    } else {
        double e[3];
        const double q2 = sep64<D>(G, x, n, i, j, e);
#pragma unroll
        for (int a = 0; a < D; ++a) d[a] = (T)e[a];
        r2 = (T)q2;
    }
}

// Cell shift of a list entry.
__device__ __forceinline__ void decode_shift(int code, int &dx, int &dy, int &dz)
{
    dx = code % 3 - 1;
    dy = (code / 3) % 3 - 1;
    dz = code / 9 - 1;
}

// The cell of a position along one axis; outside a closed axis: flagged, clamped.
__device__ __forceinline__ int cell_coord(double xa, double lo, double hi, double inv_s, int nc, int periodic,
                                          uint32_t *err)
{
    int k = (int)floor((xa - lo) * inv_s);
    if (k < 0) {
        if (!periodic && xa < lo) atomicOr(err, kErrDomain);
        k = 0;
    }
    if (k >= nc) {
        if (!periodic && xa > hi) atomicOr(err, kErrDomain);
        k = nc - 1;
    }
    return k;
}

// Counts particle i of the source order, at x, into its cell (global index).
__device__ __forceinline__ void count_key(const Buffers &B, const Geom &G, int cell_off, int i, const double *x)
{
    int c = cell_off, mult = 1;
    for (int a = 0; a < G.dim; ++a) {
        c += cell_coord(x[a], G.lo[a], G.hi[a], G.inv_s[a], G.nc[a], G.periodic[a], B.err) * mult;
        mult *= G.nc[a];
    }
    B.key[i] = c;
    B.slot[i] = atomicAdd(&B.cell_count[c], 1);
}

template <typename T> struct Packed;
template <> struct Packed<double> { using type = double4_32a; };
template <> struct Packed<float> { using type = float4; };

template <typename T>
__device__ __forceinline__ const typename Packed<T>::type *nb_ptr(const Buffers &B, int buf);
template <>
__device__ __forceinline__ const double4_32a *nb_ptr<double>(const Buffers &B, int buf) { return B.nb64[buf]; }
template <>
__device__ __forceinline__ const float4 *nb_ptr<float>(const Buffers &B, int buf) { return B.nb32[buf]; }

// Copies a table entry into shared memory with the whole block (then syncs).
template <typename T>
__device__ __forceinline__ void block_copy(T &dst, const T &src)
{
    static_assert(sizeof(T) % 4 == 0, "word copy");
    for (int w = threadIdx.x; w < (int)(sizeof(T) / 4); w += blockDim.x)
        reinterpret_cast<int *>(&dst)[w] = reinterpret_cast<const int *>(&src)[w];
    __syncthreads();
}

}  // namespace dtsph
