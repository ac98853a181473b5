// The pair terms of the FP32C path, two neighbours of a particle at a time.
//
// With one neighbour at a time the kernels that sum over neighbour lists were bound
// by instruction issue (59-66% of the issue slots busy with no pipe near its peak: 111 M
// warp instructions in the state-n pass of 61^3 particles, 54 M so; 74 M and 48% of the
// slots with the lanes shared, see warp_rates32), so the arithmetic of two
// list entries runs in the packed single-precision instructions (add, sub, mul and
// fma .f32x2: two IEEE-rounded results per issue). Entries 2m and 2m + 1 of a list
// form pair m; the even and the odd entries have their own Kahan-compensated sums,
// merged at the end with an error-free two-sum. The first operation on gathered
// values (a difference with the particle's own value) stays scalar: its result
// register can be any half of a packed operand, where packing loaded values
// costs a move each.
//
// Constants common to every pair are factored out of the sums: with dW/dr =
// (sigma / h) w(q), the cached or recomputed coefficients are g = w r_ij / r and
// F = w r / (r^2 + eta h^2), and the sums
//   S_p = sum V_ij . g + (c_edac / c_div) p_ij F
//   S_V = sum -(p_i + p_j) g + (c_visc / c_p) F V_ij
// give dp/dtau = c_div sigma/h S_p and F_i = c_p sigma/h S_V.
//
// List rows are filled up to a multiple of four with entries of the particle
// itself: r = 0 there, so g = F = 0 and they add exact zeros without a test.
#pragma once

#include "bulk.cuh"
#include "f32x2.cuh"
#include "geometry.cuh"

namespace dtsph {

// 1 / sqrt(x) and 1 / x by the special-function unit (about one ulp), x a normal
// number: without the scaling steps for subnormal arguments.
__device__ __forceinline__ float rsqrt_fast(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two Kahan sums side by side. nc is the compensation with its sign turned, so
// that the next term's first fma takes it up: add() gets the term with nc already
// in it, and the sum is s + nc.
struct Kahan2 {
    F2 s, nc;
    __device__ __forceinline__ Kahan2() : s(both(0.f)), nc(both(0.f)) {}
    __device__ __forceinline__ void add(F2 y)
    {
        const F2 t = add2(s, y);
        nc = sub2(y, sub2(t, s));
        s = t;
    }
    __device__ __forceinline__ Kahan merged() const
    {
        float s0, s1, c0, c1;
        unpack2(s, s0, s1);
        unpack2(nc, c0, c1);
        Kahan k;
        k.s = s0;
        k.c = -c0;
        k.merge(s1, -c1);
        return k;
    }
};

template <int D>
struct Sums32 {
    Kahan2 ap, F[D];
};

// g = w r_ij / r and F = w r / (r^2 + eta h^2) of two neighbours, w the quintic
// spline's dW/dq without sigma (0 from q = 3 on). 1e-37 beside r^2 leaves it as it
// is but for r = 0, where d = 0 times a finite factor and w(0) = 0 give zeros.
template <int D>
__device__ __forceinline__ void grad2(const PairK32 &k, const F2 *d, F2 *g, F2 &F)
{
    F2 r2 = fma2(d[1], d[1], fma2(d[0], d[0], both(1e-37f)));
    if (D == 3) r2 = fma2(d[2], d[2], r2);
    float ra, rb;
    unpack2(r2, ra, rb);
    const F2 rinv = pack2(rsqrt_fast(ra), rsqrt_fast(rb));
    const F2 r = mul2(r2, rinv);
    const F2 q = mul2(r, both(k.inv_h));
    float qa, qb;
    unpack2(q, qa, qb);
    const F2 a = pack2(fmaxf(__fsub_rn(3.f, qa), 0.f), fmaxf(__fsub_rn(3.f, qb), 0.f));
    const F2 b = pack2(fmaxf(__fsub_rn(2.f, qa), 0.f), fmaxf(__fsub_rn(2.f, qb), 0.f));
    const F2 c = pack2(fmaxf(__fsub_rn(1.f, qa), 0.f), fmaxf(__fsub_rn(1.f, qb), 0.f));
    const F2 a2 = mul2(a, a), b2 = mul2(b, b), c2 = mul2(c, c);
    F2 w = mul2(mul2(both(-5.f), a2), a2);
    w = fma2(mul2(both(30.f), b2), b2, w);
    w = fma2(mul2(both(-75.f), c2), c2, w);
    const F2 wr = mul2(w, rinv);
#pragma unroll
    for (int e = 0; e < D; ++e) g[e] = mul2(wr, d[e]);
    float da, db;
    unpack2(add2(r2, both(k.eta_h2)), da, db);
    F = mul2(mul2(w, r), pack2(rcp_fast(da), rcp_fast(db)));
}

// What particles moving in pseudo-time add (Eqs. dp-dtau, discrete_ME): their
// pseudo-velocity t and sum -(p_i + p_j) g; NoMove for particles fixed in it.
template <int D>
struct Move32 {
    static constexpr bool on = true;
    float t[3];
    Kahan2 np[D];
};
struct NoMove {
    static constexpr bool on = false;
};

// The contribution of two neighbours with states qa and qb (V, p) to the sums.
// WALLS: wa, wb are their velocities in the divergence term (a wall's prescribed
// one), the states' being those of the viscous terms (a wall's ghost velocity).
template <int D, bool WALLS, typename M>
__device__ __forceinline__ void pair2_accumulate(const PairK32 &k, const F2 *g, F2 F, const float *vi, float pi,
                                                 float4 qa, float4 qb, const float *wa, const float *wb,
                                                 Sums32<D> &A, M &mv)
{
    const float va[3] = {qa.x, qa.y, qa.z}, vb[3] = {qb.x, qb.y, qb.z};
    F2 dv[D];
    F2 y = A.ap.nc;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        dv[a] = pack2(__fsub_rn(vi[a], va[a]), __fsub_rn(vi[a], vb[a]));
        if constexpr (WALLS) y = fma2(pack2(__fsub_rn(vi[a], wa[a]), __fsub_rn(vi[a], wb[a])), g[a], y);
        else y = fma2(dv[a], g[a], y);
    }
    const F2 dp = pack2(__fsub_rn(pi, qa.w), __fsub_rn(pi, qb.w));
    A.ap.add(fma2(mul2(both(k.ed), dp), F, y));
    F2 np = pack2(__fsub_rn(-pi, qa.w), __fsub_rn(-pi, qb.w));    // -(p_i + p_j)
    F2 conv = both(0.f);
    if constexpr (M::on) {
        // advection: (V_i + V_j) m/rho0 (V~_i . g), and the pressure sum that V~_i meets
        conv = mul2(both(mv.t[0]), g[0]);
#pragma unroll
        for (int a = 1; a < D; ++a) conv = fma2(both(mv.t[a]), g[a], conv);
        conv = mul2(both(k.vol), conv);
#pragma unroll
        for (int a = 0; a < D; ++a) mv.np[a].add(fma2(np, g[a], mv.np[a].nc));
    }
    // the terms that most runs do without (artificial viscosity, the steady-mode
    // convection) sit behind one uniform test
    if (k.rare) {
        if (k.use_av) {
            // v_ij . r_ij < 0  <=>  v_ij . g > 0 (w < 0); -m Pi_ij
            F2 vg = mul2(dv[0], g[0]), g2 = mul2(g[0], g[0]);
#pragma unroll
            for (int a = 1; a < D; ++a) {
                vg = fma2(dv[a], g[a], vg);
                g2 = fma2(g[a], g[a], g2);
            }
            float v0, v1, s0, s1, f0, f1, p0, p1;
            unpack2(vg, v0, v1);
            unpack2(g2, s0, s1);
            unpack2(F, f0, f1);
            unpack2(np, p0, p1);
            if (v0 > 0.f && s0 > 0.f) p0 = __fadd_rn(p0, __fmul_rn(k.av, __fmul_rn(v0, f0)) / s0);
            if (v1 > 0.f && s1 > 0.f) p1 = __fadd_rn(p1, __fmul_rn(k.av, __fmul_rn(v1, f1)) / s1);
            np = pack2(p0, p1);
        }
        if (k.steady) {
            // convection of Eq. (mom-steady): -(V_i + V_j) m/rho0 (V_i . g)
            conv = mul2(both(vi[0]), g[0]);
#pragma unroll
            for (int a = 1; a < D; ++a) conv = fma2(both(vi[a]), g[a], conv);
            conv = mul2(both(-k.vol), conv);
        }
    }
    const F2 cv = mul2(both(k.visc), F);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        F2 z = fma2(cv, dv[a], fma2(np, g[a], A.F[a].nc));
        if (M::on || (k.rare && k.steady))
            z = fma2(conv, WALLS ? pack2(__fadd_rn(vi[a], wa[a]), __fadd_rn(vi[a], wb[a]))
                                 : pack2(__fadd_rn(vi[a], va[a]), __fadd_rn(vi[a], vb[a])), z);
        A.F[a].add(z);
    }
}

// A sum's even and odd halves merged, then the particle's L lanes.
template <int L>
__device__ __forceinline__ float merged32(const Kahan2 &a)
{
    Kahan m = a.merged();
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) m.shfl_merge(o);
    return m.value();
}

// The rates with their factors.
template <int D, int L>
__device__ __forceinline__ void rates32(const PairK32 &k, const Sums32<D> &A, float &ap, float *F)
{
    ap = __fmul_rn(k.s_ap, merged32<L>(A.ap));
#pragma unroll
    for (int a = 0; a < D; ++a) F[a] = __fmul_rn(k.s_F, merged32<L>(A.F[a]));
}

// Displacement of the home offset for every shift code, by component, in shared
// memory: o_i moves by minus the cell shift (a particle's own code, 13, by zero). The
// codes of a warp's entries differ, and 32 words by component lie in 32 banks: one
// wavefront a component (records of 16 bytes: 2.5% more time in the 128^3 loop
// without the cache).
constexpr int kCodes = 32;
struct ShiftTable {
    float c[3][kCodes];
};
__device__ __forceinline__ void load_shifts(ShiftTable &sh, const Geom &G)     // (whole block; sync after)
{
    const int code = threadIdx.x;
    if (code >= kCodes) return;
    int dx, dy, dz;
    decode_shift(code < 27 ? code : 13, dx, dy, dz);
    sh.c[0][code] = -(float)dx * G.s_f[0];
    sh.c[1][code] = -(float)dy * G.s_f[1];
    sh.c[2][code] = -(float)dz * G.s_f[2];
}

// r_ij of list entry e: (o_i - shift) - o_j.
template <int D>
__device__ __forceinline__ void entry_sep(const ShiftTable &sh, float4 oi, float4 oj, uint32_t e, float *d)
{
    const int t = entry_code(e);
    d[0] = __fsub_rn(__fadd_rn(oi.x, sh.c[0][t]), oj.x);
    d[1] = __fsub_rn(__fadd_rn(oi.y, sh.c[1][t]), oj.y);
    if (D == 3) d[2] = __fsub_rn(__fadd_rn(oi.z, sh.c[2][t]), oj.z);
}

// g and F of list entries ea, eb with the neighbours' offsets oa, ob.
template <int D>
__device__ __forceinline__ void entry_grad2(const PairK32 &k, const ShiftTable &sh, float4 oi, float4 oa, float4 ob,
                                            uint32_t ea, uint32_t eb, F2 *g, F2 &F)
{
    float da[3], db[3];
    entry_sep<D>(sh, oi, oa, ea, da);
    entry_sep<D>(sh, oi, ob, eb, db);
    F2 d[D];
#pragma unroll
    for (int a = 0; a < D; ++a) d[a] = pack2(da[a], db[a]);
    grad2<D>(k, d, g, F);
}

// Pairs of a list of cnt entries, the fill up to a multiple of four included.
__host__ __device__ __forceinline__ int list_pairs(int cnt) { return (cnt + 3) / 4 * 2; }

// The sums over the list lst of a particle by L lanes (lane_in takes the pairs
// lane_in, lane_in + L, ..., two in flight): offsets off, states nb, geometry
// recomputed. wall(entry, w) gives a neighbour's divergence-term velocity (WALLS).
template <int D, bool WALLS, int L, typename WV, typename M>
__device__ __forceinline__ void list_sums32(const PairK32 &k, const ShiftTable &sh, const uint32_t *__restrict__ lst,
                                            int cnt, int lane_in, float4 oi, const float *vi, float pi,
                                            const float4 *off, const float4 *nb, WV wall, Sums32<D> &A, M &mv)
{
    const int np = list_pairs(cnt);
    for (int m = lane_in; m < np; m += 2 * L) {
        uint32_t e[4];
        const bool two = L == 1 || m + L < np;      // (one lane: the pairs come in twos)
        if constexpr (L == 1) {
            const uint4 v = *reinterpret_cast<const uint4 *>(lst + 2 * m);
            e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
        } else {
            const uint2 v = *reinterpret_cast<const uint2 *>(lst + 2 * m);
            const uint2 u = *reinterpret_cast<const uint2 *>(lst + 2 * (two ? m + L : m));
            e[0] = v.x; e[1] = v.y; e[2] = u.x; e[3] = u.y;
        }
        float4 o[4], q[4];
        float w[4][3];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int j = entry_slot(e[r]);
            o[r] = off[j];
            q[r] = nb[j];
            if constexpr (WALLS) wall(e[r], q[r], w[r]);
        }
#pragma unroll
        for (int r = 0; r < 4; r += 2) {
            if (r == 2 && !two) break;
            F2 g[D], F;
            entry_grad2<D>(k, sh, oi, o[r], o[r + 1], e[r], e[r + 1], g, F);
            pair2_accumulate<D, WALLS>(k, g, F, vi, pi, q[r], q[r + 1], w[r], w[r + 1], A, mv);
        }
    }
}

// The rates of a warp's 32 slots (s: the lane's own, cnt its list's length, 0 if it
// has no rates to form), G lanes to a slot: the warp takes 32 / G slots at a time,
// so that a gather's 32 entries are G neighbours in a row of each of them and fall
// on fewer lines: the L1 looks up one line a cycle. Tag lookups a load, by counter at
// 61^3: 17.5 with one lane per slot (the loop without the cache), 8.3 with eight. A slot's sums then come back to its own lane. sums(slot, lane of the slot,
// count, V_i, p_i, A) adds the pairs.
template <int D, int G, typename SUMS>
__device__ __forceinline__ void warp_rates32(const PairK32 &k, int s, int cnt, const float4 *nb, SUMS sums, float &ap,
                                             float *F)
{
    constexpr int P = kWarp / G;                         // slots at a time
    const int lane = threadIdx.x & (kWarp - 1), s0 = s - lane;
    ap = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a] = 0.f;
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
        const int from = g * P + lane / G;               // the slot this lane works on
        const int c = __shfl_sync(0xffffffffu, cnt, from), sg = s0 + from;
        const float4 qi = c > 0 ? nb[sg] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float vi[3] = {qi.x, qi.y, qi.z};
        Sums32<D> A;
        sums(sg, lane % G, c, vi, qi.w, A);
        float r[D + 1];
        rates32<D, G>(k, A, r[0], r + 1);
        const int src = (lane - g * P) * G & (kWarp - 1);
        const bool mine = lane / P == g;
#pragma unroll
        for (int a = 0; a <= D; ++a) {
            const float v = __shfl_sync(0xffffffffu, r[a], src);
            if (mine) (a == 0 ? ap : F[a - 1]) = v;
        }
    }
}

// ------------------------------------------------------------ the pair cache
//
// FP32C records hold two list entries (a pair m of a slot): two float4, (g_x, g_x',
// g_y, g_y') and in 2D (F, F', entry, entry'), in 3D (g_z, g_z', F, F') with the
// entries as a uint2 in pj; an entry is the neighbour's slot and its wall flag. For
// a wall slot the coefficients are (W, W', Wg, Wg'). Sliced by warp: pair m of slot
// s is row (s / 32) cache_rows(K) + m, its two float4 32 records apart, so a warp
// reads and writes whole 512-byte rows.
__host__ __device__ constexpr int cache_rows(int K) { return (K + 3) / 4 * 2; }

struct CachePair {
    float4 c0, c1;
    uint32_t ea, eb;
};

template <int D>
__device__ __forceinline__ void cache_coefs(const CachePair &r, F2 *g, F2 &F)
{
    g[0] = pack2(r.c0.x, r.c0.y);
    g[1] = pack2(r.c0.z, r.c0.w);
    if constexpr (D == 3) {
        g[2] = pack2(r.c1.x, r.c1.y);
        F = pack2(r.c1.z, r.c1.w);
    } else {
        F = pack2(r.c1.x, r.c1.y);
    }
}

// First row of slot s's slice.
__device__ __forceinline__ size_t cache_row(const Buffers &B, int s)
{
    return (size_t)(s >> 5) * cache_rows(B.K);
}

// The record of lane `lane` (slot % 32) in a row.
template <int D>
__device__ __forceinline__ CachePair cache_pair(const Buffers &B, size_t row, int lane)
{
    const float4 *p = B.pc32 + row * 2 * kWarp + lane;
    CachePair r;
    r.c0 = p[0];
    r.c1 = p[kWarp];
    if constexpr (D == 3) {
        const uint2 e = reinterpret_cast<const uint2 *>(B.pj)[row * kWarp + lane];
        r.ea = e.x;
        r.eb = e.y;
    } else {
        r.ea = __float_as_uint(r.c1.z);
        r.eb = __float_as_uint(r.c1.w);
    }
    return r;
}

// The same for rows read once per pass, not kept in L1.
template <int D>
__device__ __forceinline__ CachePair cache_pair_stream(const Buffers &B, size_t row, int lane, uint64_t policy)
{
    const float4 *p = B.pc32 + row * 2 * kWarp + lane;
    CachePair r;
    r.c0 = ld_f4_stream(p, policy);
    r.c1 = ld_f4_stream(p + kWarp, policy);
    if constexpr (D == 3) {
        const uint2 e = ld_u2_stream(reinterpret_cast<const uint2 *>(B.pj) + row * kWarp + lane, policy);
        r.ea = e.x;
        r.eb = e.y;
    } else {
        r.ea = __float_as_uint(r.c1.z);
        r.eb = __float_as_uint(r.c1.w);
    }
    return r;
}

}  // namespace dtsph
