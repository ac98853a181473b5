// The kernels that walk the neighbour lists (built in lists.cu): the wall
// extrapolation and the pair pass at the state n, the pair-coefficient cache
// that the pseudo-time loop reads (geometry frozen for the whole loop, Sec. 2.2;
// caching kernel gradients across pseudo-iterations is the speed-up the paper
// points at in Sec. 4.7 but did not implement), and particle shifting. The
// lists hold only pairs within the cutoff, so the pair arithmetic never runs
// under the distance test, which most candidates fail.
#include "geometry.cuh"
#include "loop_rules.cuh"
#include "pair32.cuh"
#include "pair64.cuh"

namespace dtsph {

namespace {

// ---------------------------------------------------------------- walls, state n

// The list walkers below give each slot a group of L lanes; lane l of a group
// takes the list entries (FP32C: pairs of entries) l, l + L, ... Summing kernels
// merge the lanes' partial sums by shuffles, so their summation order depends on L
// alone: they use a fixed L per path, which keeps every context (solo or batched,
// any size) on the same order. FP32C: one lane per slot, the warp sharing the slots'
// lists inside (kStateLanes). FP64: eight, a small problem's chain of
// pairs being what its pass takes (1,024 2D particles: 139 us with one lane, 14 us
// now, the factored sums included), at no cost to large ones, which the FP64
// pipe bounds. Block b covers slots b * (kBlock / L) ...

template <bool F32>
constexpr int kSumLanes = F32 ? 1 : 8;
// Lanes a slot within the warp in the FP32C state-n pass (warp_rates32). 128^3: one
// lane 1.1 ms a pass, eight 0.78 ms; in 2D four take 1% off a step of the 64-vortex
// batch and of the 200 x 200 vortex. (In the loops, whose iterations find the
// states in no L1, lanes sharing a warp's slots measured slower: 128^3 without the
// cache 1.23 ms an iteration at one lane, 1.48 at eight.)
template <int D>
constexpr int kStateLanes = D == 3 ? 8 : 4;

// Adami et al. wall values at state n in order B: p_w = (sum_f p_f W + rho0 g .
// sum_f r_wf W) / sum_f W, ghost velocity 2 v_w - sum_f V_f W / sum_f W; written
// into the packed (V, p) of the wall slot, from its neighbour list at r^n.
template <int D, bool F32, int L>
__global__ void __launch_bounds__(kBlock) k_walls_state_n(Buffers B)
{
    grid_start<false>();
    using T = typename std::conditional<F32, float, double>::type;
    constexpr int SPB = kBlock / L;
    __shared__ Geom G;
    __shared__ Phys P;
    const int inst = block_instance(B, blockIdx.x * SPB);
    block_copy(G, B.geo[inst]);
    block_copy(P, B.phys[inst]);
    const int s = blockIdx.x * SPB + threadIdx.x / L, lane_in = threadIdx.x % L;
    // every lane stays to the end: the partial sums are merged by full-warp shuffles
    const uint32_t gs = s < B.n ? B.gid_b[s] : kNoParticle;
    const bool wall = gs != kNoParticle && gs >= (uint32_t)B.nf;
    const auto *nb = nb_ptr<T>(B, 1);
    const float4 oi = wall && F32 ? B.off[s] : make_float4(0, 0, 0, 0);
    double acc[6] = {0, 0, 0, 0, 0, 0};   // sum W, sum p W, sum rho0 (g . r) W, sum V W
    const double sigma = P.sig_h * P.h;
    const uint32_t *lst = slot_list(B, s);
    const int cnt = wall ? B.pcount[s] : 0;
    for (int k = lane_in; k < cnt; k += L) {
        const uint32_t jb = lst[k];
        if (jb & kWallBit) continue;                    // fluid neighbours only
        const int j = entry_slot(jb);
        int dx, dy, dz;
        decode_shift(entry_code(jb), dx, dy, dz);
        T d[3], r2;
        listed_sep<D, F32, T>(G, B.x_b, B.off, B.n, s, j, oi, dx, dy, dz, d, r2);
        const double W = sigma * (double)quintic_w<T>(Ar<T>::mul(sqrt(r2), (T)P.inv_h));
        const auto q = nb[j];
        double gr = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) gr += P.g[a] * (double)d[a];
        acc[0] += W;
        acc[1] += (double)q.w * W;
        acc[2] += P.rho0 * gr * W;
        acc[3] += (double)q.x * W;
        acc[4] += (double)q.y * W;
        acc[5] += (double)q.z * W;
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
        for (int t = 0; t < 6; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], o);
    if (!wall || lane_in != 0) return;
    const double sw = acc[0];
    double gv[3];
    for (int a = 0; a < 3; ++a) {
        const double vw = a < D ? B.vn_b[(size_t)a * B.n + s] : 0.0;
        gv[a] = 2.0 * vw - (sw > 0 ? acc[3 + a] / sw : 0.0);
    }
    double pw = sw > 0 ? (acc[1] + acc[2]) / sw : 0.0;
    if (pw < 0.0 && P.free_surface) pw = 0.0;     // free-surface runs keep it >= 0 (Sec. 3.2)
    if (F32) B.nb32[1][s] = make_float4((float)gv[0], (float)gv[1], (float)gv[2], (float)pw);
    else B.nb64[1][s] = make_double4_32a(gv[0], gv[1], gv[2], pw);
}

// ------------------------------------------------------------------ state n pass

// Rates at (r^n, V^n, p^n) in order B over the neighbour lists at r^n. With
// PRED, also the predictor of Eqs. (v0, r0): V^0 = V^n + dt F^n, r^0 = r^n +
// dt V^n + dt^2/2 F^n; the first pressure half step p-hat^0 = p^n + dtau/2
// dp^n/dtau (Eq. pkstar_frozen with the state-n rate); and the BDF2 source
// (V^{n-1} - 4 V^n) / (2 dt) of Eq. (dv_dtau_exact), all in FP64.
template <int D, bool F32, bool PRED, bool WALLS, int L>
__global__ void __launch_bounds__(kBlock, F32 ? (D == 2 ? 4 : 3) : 1) k_state_n(Buffers B)
{
    grid_start<false>();
    using T = typename std::conditional<F32, float, double>::type;
    constexpr int SPB = kBlock / L;
    __shared__ Geom G;
    __shared__ Phys P;
    __shared__ ShiftTable sh;
    const int inst = block_instance(B, blockIdx.x * SPB);
    if (F32) load_shifts(sh, B.geo[inst]);
    block_copy(G, B.geo[inst]);
    block_copy(P, B.phys[inst]);
    const int n = B.n;
    const int s = blockIdx.x * SPB + threadIdx.x / L, lane_in = threadIdx.x % L;
    // every lane stays to the end: the partial sums are merged by full-warp shuffles
    const uint32_t gs = s < n ? B.gid_b[s] : kNoParticle;
    const bool fluid = gs < (uint32_t)B.nf;
    T apT = T(0), FT[3] = {T(0), T(0), T(0)};
    const int cnt = fluid ? B.pcount[s] : 0;
    const uint32_t *lst = slot_list(B, s);
    if constexpr (F32) {
        static_assert(L == 1, "a warp's lanes and slots one to one");
        const PairK32 k = P.k32;
        const float4 *nb = B.nb32[1];
        auto wall = [&](uint32_t e, const float4 &q, float *w) {
            w[0] = q.x; w[1] = q.y; w[2] = q.z;
            if (e & kWallBit)
                for (int a = 0; a < D; ++a) w[a] = (float)B.vn_b[(size_t)a * n + entry_slot(e)];
        };
        constexpr int G = kStateLanes<D>;
        warp_rates32<D, G>(
            k, s, cnt, nb,
            [&](int sg, int sub, int c, const float *vi, float pi, Sums32<D> &A) {
                const float4 oi = c > 0 ? B.off[sg] : make_float4(0.f, 0.f, 0.f, 0.f);
                NoMove mv;
                list_sums32<D, WALLS, G>(k, sh, slot_list(B, sg), c, sub, oi, vi, pi, B.off, nb, wall, A, mv);
            },
            apT, FT);
    } else {
        const double4_32a *nb = B.nb64[1];
        const PairConst<double> k = pair_const<double>(P);
        Sums64<D> A;
        double xi[3] = {0, 0, 0};
        if (fluid)
            for (int a = 0; a < D; ++a) xi[a] = B.x_b[(size_t)a * n + s];
        const double4_32a qi = fluid ? nb[s] : make_double4_32a(0, 0, 0, 0);
        const double vi[3] = {qi.x, qi.y, qi.z};
        // R entries per round: their indices, then their gathers, then the pair
        // terms, so that R loads are in flight per lane; the entries keep their order
        constexpr int R = 4;
        for (int q0 = lane_in; q0 < cnt; q0 += L * R) {
            uint32_t jbv[R];
            double4_32a qv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) jbv[r] = lst[min(q0 + r * L, cnt - 1)];
#pragma unroll
            for (int r = 0; r < R; ++r) qv[r] = nb[entry_slot(jbv[r])];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (q0 + r * L >= cnt) break;
                const int j = entry_slot(jbv[r]);
                double d[3], g[3], F;
                const double r2 = listed_sep64<D>(G, xi, B.x_b, n, j, d);
                grad64<D>(P, d, r2, g, F);
                const double vv[3] = {qv[r].x, qv[r].y, qv[r].z};
                if constexpr (WALLS) {
                    double vd[3] = {vv[0], vv[1], vv[2]};
                    if (jbv[r] & kWallBit)
                        for (int a = 0; a < D; ++a) vd[a] = B.vn_b[(size_t)a * n + j];
                    pair64_accumulate<D, true>(k, g, F, vi, qi.w, vd, vv, qv[r].w, A);
                } else {
                    pair64_accumulate<D, false>(k, g, F, vi, qi.w, vv, vv, qv[r].w, A);
                }
            }
        }
        rates64<D, L>(P, k, A, apT, FT);
    }
    if (lane_in != 0) return;
    if (gs == kNoParticle) {
        if (PRED && s < n) B.key[s] = -1;
        return;
    }
    double xp[3] = {0, 0, 0};                        // r^0
    if (!fluid) {
        if (PRED) {
            for (int a = 0; a < D; ++a) B.xp_b[(size_t)a * n + s] = xp[a] = B.x_b[(size_t)a * n + s];
            count_key(B, G, B.inst[inst].cell_off, s, xp);
        }
        return;
    }
    const double apv = (double)apT;
    double Fv[3];
    for (int a = 0; a < D; ++a) Fv[a] = __dadd_rn((double)FT[a], P.g[a]);
    B.ap_b[s] = apv;
    for (int a = 0; a < D; ++a) B.f_b[(size_t)a * n + s] = Fv[a];
    if (PRED && P.steady) {
        // steady mode: the iteration starts from the state itself, the particles
        // stay, and the source is -g (the loop forms F + g - 0)
        for (int a = 0; a < D; ++a) {
            const size_t q = (size_t)a * n + s;
            B.xp_b[q] = xp[a] = B.x_b[q];
            B.v0_b[q] = B.vn_b[q];
            B.s_b[q] = -P.g[a];
        }
        B.ph0_b[s] = __fma_rn(0.5 * P.dtau, apv, B.pn_b[s]);
    } else if (PRED) {
        for (int a = 0; a < D; ++a) {
            const size_t q = (size_t)a * n + s;
            // explicit roundings: the same bits in every kernel variant
            const double V = B.vn_b[q];
            xp[a] = __fma_rn(0.5 * P.dt * P.dt, Fv[a], __fma_rn(P.dt, V, B.x_b[q]));
            if (G.periodic[a]) {
                if (xp[a] >= G.hi[a]) xp[a] = __dsub_rn(xp[a], G.L[a]);
                else if (xp[a] < G.lo[a]) xp[a] = __dadd_rn(xp[a], G.L[a]);
            }
            B.xp_b[q] = xp[a];
            B.v0_b[q] = __fma_rn(P.dt, Fv[a], V);
            B.s_b[q] = __dmul_rn(P.kappa, __fma_rn(__fma_rn(-4.0, V, B.vnm1_b[q]), P.inv_2dt, -P.g[a]));
        }
        B.ph0_b[s] = __fma_rn(0.5 * P.dtau, apv, B.pn_b[s]);
    }
    if (PRED) count_key(B, G, B.inst[inst].cell_off, s, xp);     // for the binning at r^0
}

// --------------------------------------------------------------- pair cache

// The cache records of slot s (its list, in the sliced layout), FP32C: lane
// threadIdx.x % L of the slot's group takes the pairs of entries lane, lane + L, ...,
// two in flight.
template <int D, int L>
__device__ __forceinline__ void pair_cache_slot32(const Buffers &B, const Phys &P, const ShiftTable &sh,
                                                  const uint32_t *__restrict__ gid, int s)
{
    const PairK32 k = P.k32;
    const bool wall_s = gid[s] >= (uint32_t)B.nf;
    const uint32_t *lst = slot_list(B, s);
    const size_t row0 = cache_row(B, s);
    const float4 oi = B.off[s];
    const int np = list_pairs(B.pcount[s]);
    auto put = [&](int m, uint32_t ea, uint32_t eb, float4 oa, float4 ob) {
        CachePair c;
        if (wall_s) {
            // (a wall row's fill holds W(0); the wall values count the list's entries only)
            float W[2], Wg[2];
            const float sigma = (float)(P.sig_h * P.h);
            const uint32_t e[2] = {ea, eb};
            const float4 o[2] = {oa, ob};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float d[3];
                entry_sep<D>(sh, oi, o[i], e[i], d);
                float r2 = __fmaf_rn(d[1], d[1], __fmul_rn(d[0], d[0]));
                if (D == 3) r2 = __fmaf_rn(d[2], d[2], r2);
                W[i] = __fmul_rn(sigma, quintic_w<float>(__fmul_rn(sqrtf(r2), k.inv_h)));
                float gr = 0.f;
                for (int a = 0; a < D; ++a) gr += (float)P.g[a] * d[a];
                Wg[i] = (float)P.rho0 * gr * W[i];
            }
            c.c0 = make_float4(W[0], W[1], Wg[0], Wg[1]);
            c.c1 = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            F2 g[D], F;
            entry_grad2<D>(k, sh, oi, oa, ob, ea, eb, g, F);
            unpack2(g[0], c.c0.x, c.c0.y);
            unpack2(g[1], c.c0.z, c.c0.w);
            if constexpr (D == 3) {
                unpack2(g[2], c.c1.x, c.c1.y);
                unpack2(F, c.c1.z, c.c1.w);
            } else {
                unpack2(F, c.c1.x, c.c1.y);
            }
        }
        const uint32_t ja = ea & ~kCodeMask, jb = eb & ~kCodeMask;      // what the pseudo-time loop reads
        float4 *p = B.pc32 + (row0 + m) * 2 * kWarp + (s & 31);
        if constexpr (D == 3) {
            reinterpret_cast<uint2 *>(B.pj)[(row0 + m) * kWarp + (s & 31)] = make_uint2(ja, jb);
        } else {
            c.c1.z = __uint_as_float(ja);
            c.c1.w = __uint_as_float(jb);
        }
        p[0] = c.c0;
        p[kWarp] = c.c1;
    };
    for (int m = threadIdx.x % L; m < np; m += 2 * L) {
        const bool two = L == 1 || m + L < np;          // (one lane: the pairs come in twos)
        uint32_t e[4];
        if constexpr (L == 1) {
            const uint4 v = *reinterpret_cast<const uint4 *>(lst + 2 * m);
            e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
        } else {
            const uint2 v = *reinterpret_cast<const uint2 *>(lst + 2 * m);
            const uint2 u = *reinterpret_cast<const uint2 *>(lst + 2 * (two ? m + L : m));
            e[0] = v.x; e[1] = v.y; e[2] = u.x; e[3] = u.y;
        }
        float4 o[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) o[r] = B.off[entry_slot(e[r])];
        put(m, e[0], e[1], o[0], o[1]);
        if (two) put(m + L, e[2], e[3], o[2], o[3]);
    }
}

// The same for FP64, entry by entry.
template <int D, int L>
__device__ __forceinline__ void pair_cache_slot64(const Buffers &B, const Geom &G, const Phys &P,
                                                  const double *__restrict__ xpos, const uint32_t *__restrict__ gid,
                                                  int s)
{
    const bool wall_s = gid[s] >= (uint32_t)B.nf;
    const uint32_t *lst = slot_list(B, s);                           // the list, per slot
    const size_t base = (size_t)(s >> 5) * B.K * kWarp + (s & 31);   // the cache rows, sliced
    const double sigma = P.sig_h * P.h;
    const int cnt = B.pcount[s];
    double xi[3] = {0, 0, 0};
    for (int a = 0; a < D; ++a) xi[a] = xpos[(size_t)a * B.n + s];
    for (int q = threadIdx.x % L; q < cnt; q += L) {
        const size_t e = base + (size_t)q * kWarp;
        const uint32_t jb = lst[q] & ~kCodeMask;      // what the pseudo-time loop reads
        double d[3], g[3] = {0, 0, 0}, F = 0;
        const double r2 = listed_sep64<D>(G, xi, xpos, B.n, entry_slot(jb), d);
        if (wall_s) {
            const double W = Ar<double>::mul(sigma, quintic_w<double>(Ar<double>::mul(sqrt(r2), P.inv_h)));
            double gr = 0;
            for (int a = 0; a < D; ++a) gr += P.g[a] * d[a];
            g[0] = W;
            g[1] = P.rho0 * gr * W;
        } else {
            // layout (g, F)
            grad64<D>(P, d, r2, g, F);
        }
        B.pc64[e] = make_double4_32a(g[0], g[1], D == 3 && !wall_s ? g[2] : 0.0, F);
        B.pj[e] = jb;
    }
}

// The pair coefficients of every list entry (order of the latest binning):
// gradW_ij and F_ij for a fluid slot, W_wf and rho0 (g . r_wf) W_wf for a wall
// slot, at the entry's place in the sliced layout. Entries are independent, so
// L only sets the parallelism.
template <int D, bool F32, int L>
__global__ void __launch_bounds__(kBlock) k_pair_cache(Buffers B, const double *__restrict__ xpos,
                                                       const uint32_t *__restrict__ gid)
{
    constexpr int SPB = kBlock / L;
    __shared__ Geom G;
    __shared__ Phys P;
    __shared__ ShiftTable sh;
    if (skip_form(B)) return;            // the step runs the other pair-term form
    // tiles of SPB slots, grid-stride (a launch with one block per tile takes
    // one each; a launch in a graph that may skip it takes one wave of blocks,
    // so that skipping costs little)
    const int ntile = (B.n + SPB - 1) / SPB;
    int p_inst = -1;
    for (int bt = blockIdx.x; bt < ntile; bt += gridDim.x) {
        const int inst = block_instance(B, bt * SPB);
        if (inst != p_inst) {
            __syncthreads();                 // the previous tile is done with G and P
            if (F32) load_shifts(sh, B.geo[inst]);
            block_copy(G, B.geo[inst]);
            block_copy(P, B.phys[inst]);
            p_inst = inst;
        }
        const int s = bt * SPB + threadIdx.x / L;
        if (s < B.n && gid[s] != kNoParticle) {
            if constexpr (F32) pair_cache_slot32<D, L>(B, P, sh, gid, s);
            else pair_cache_slot64<D, L>(B, G, P, xpos, gid, s);
        }
    }
}

// ---------------------------------------------------------------- shifting

// Particle shifting after the real step (Sec. 3.5), in order B at r^{n+1}, one
// lane per slot; the displacement over every neighbour (wall particles continue
// the particle distribution), the gradients of the correction over fluid
// neighbours (free-surface runs: particles with div r_i < dim - 1/2, fluid and
// wall neighbours counted, stay where they are):
//   dr_i = -(h^2/2) sum_j V_j (1 + W_ij / W(h)) gradW_ij          Eq. (shift-deltar)
//   f_i <- f_i + (grad f)_i . dr_i, (grad f)_i = sum_j V_j (f_j - f_i) gradW_ij
//                                                      for f = p, V   Eq. (shift-correct)
//   r_i <- r_i + dr_i (wrapped on periodic axes)
// with V_j = m / rho0 and W(h) the kernel at r = h. Every gradient uses the
// unshifted fields (reads order B); the shifted r, V, p go to the particle's
// slot in order A (perm), which the next step bins again.
template <int D, bool F32>
__global__ void __launch_bounds__(kBlock) k_shift(Buffers B)
{
    using T = typename std::conditional<F32, float, double>::type;
    using Acc = typename std::conditional<F32, Kahan, Plain64>::type;
    __shared__ Geom G;
    __shared__ Phys P;
    const int inst = block_instance(B, blockIdx.x * kBlock);
    block_copy(G, B.geo[inst]);
    block_copy(P, B.phys[inst]);
    const int n = B.n;
    const int s = blockIdx.x * kBlock + threadIdx.x;
    if (s >= n) return;
    if (B.gid_b[s] >= (uint32_t)B.nf) return;            // walls and padding stay
    const auto *nb = nb_ptr<T>(B, 1);                     // (V, p) at r^{n+1}, order B
    const auto qi = nb[s];
    const T vi[3] = {(T)qi.x, (T)qi.y, (T)qi.z};
    const T pi = (T)qi.w;
    const float4 oi = F32 ? B.off[s] : make_float4(0, 0, 0, 0);
    const T vol = (T)(P.m / P.rho0);
    const T sigma = (T)(P.sig_h * P.h);
    const T w_h = sigma * quintic_w<T>(T(1));
    Acc dr[3], gp[3], gv[3][3];
    double divr = 0.0;            // div r_i = -sum_j V_j r_ij . gradW_ij, walls included
    const uint32_t *lst = slot_list(B, s);
    const int cnt = B.pcount[s];
    for (int k = 0; k < cnt; ++k) {
        const uint32_t jb = lst[k];
        const int j = entry_slot(jb);
        int dx, dy, dz;
        decode_shift(entry_code(jb), dx, dy, dz);
        T d[3], r2;
        listed_sep<D, F32, T>(G, B.x_b, B.off, n, s, j, oi, dx, dy, dz, d, r2);
        const T r = sqrt(r2);
        const T q = r * (T)P.inv_h;
        const T a = r > T(0) ? (T)P.sig_h * quintic_dwdq<T>(q) / r : T(0);
        divr -= (double)(vol * a * r2);                   // r_ij . gradW_ij = (dW/dr / r) r^2
        // the displacement counts every neighbour, wall particles included
        // (they continue the particle distribution)
        const T fdr = vol * (T(1) + sigma * quintic_w<T>(q) / w_h);
#pragma unroll
        for (int c = 0; c < D; ++c) dr[c].add(fdr * (a * d[c]));
        if (jb & kWallBit) continue;                      // the gradients: fluid neighbours only

        const auto qj = nb[j];
        const T vj[3] = {(T)qj.x, (T)qj.y, (T)qj.z};
        const T dp = vol * ((T)qj.w - pi);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const T gw = a * d[c];
            gp[c].add(dp * gw);
#pragma unroll
            for (int b2 = 0; b2 < D; ++b2) gv[b2][c].add(vol * (vj[b2] - vi[b2]) * gw);
        }
    }
    // a free-surface particle (Lind et al.'s test, Sec. 3.5) is not shifted
    const bool surface = P.free_surface && divr < (double)D - 0.5;
    const double dmul = surface ? 0.0 : -0.5 * P.h * P.h;
    double drv[3] = {0, 0, 0};
    for (int c = 0; c < D; ++c) drv[c] = dmul * (double)(T)dr[c].value();
    const int o = B.perm[s];
    double pnew = B.pn_b[s];
    for (int c = 0; c < D; ++c) pnew += (double)(T)gp[c].value() * drv[c];
    B.pn_a[o] = pnew;
    for (int b2 = 0; b2 < D; ++b2) {
        double v = B.vn_b[(size_t)b2 * n + s];
        for (int c = 0; c < D; ++c) v += (double)(T)gv[b2][c].value() * drv[c];
        B.vn_a[(size_t)b2 * n + o] = v;
        double x = B.x_b[(size_t)b2 * n + s] + drv[b2];
        if (G.periodic[b2]) {
            if (x >= G.hi[b2]) x -= G.L[b2];
            else if (x < G.lo[b2]) x += G.L[b2];
        }
        B.x_a[(size_t)b2 * n + o] = x;
    }
}

}  // namespace

// Lanes per slot of the pair-coefficient pass: enough warps to fill the GPU on
// small problems (each slot's chain of entries is latency-bound), one lane per
// slot on large ones.
int nlist_lanes(int n)
{
    int L = 1;
    while (L < 8 && (long long)n * L < 400000) L *= 2;
    return L;
}

// Neighbour lists at r^n (order B), then the wall values and the state-n pass.
int launch_state_n(const Buffers &B, bool predictor, cudaStream_t st, bool build_lists)
{
    int k = 0;
    if (build_lists) {
        launch_nlist(B, B.x_b, st);
        k = 1;
    }
    DTSPH_DISPATCH(B.dim, B.fp32c, {
        constexpr int L = kSumLanes<F32>;
        const int nb = (int)(((long long)B.n * L + kBlock - 1) / kBlock);
        if (B.nw > 0) {
            launch_next(B, st, nb, kBlock, k_walls_state_n<D, F32, L>, B);
            ++k;
            if (predictor) launch_next(B, st, nb, kBlock, k_state_n<D, F32, true, true, L>, B);
            else launch_next(B, st, nb, kBlock, k_state_n<D, F32, false, true, L>, B);
        } else if (predictor) {
            launch_next(B, st, nb, kBlock, k_state_n<D, F32, true, false, L>, B);
        } else {
            launch_next(B, st, nb, kBlock, k_state_n<D, F32, false, false, L>, B);
        }
    });
    return k + 1;
}

// Neighbour lists at xpos, then the pair coefficients.
int launch_pair_cache(const Buffers &B, const double *xpos, const uint32_t *gid, cudaStream_t st)
{
    launch_nlist(B, xpos, st);
    return 1 + launch_pair_cache_pass(B, xpos, gid, st);
}

int launch_pair_cache_pass(const Buffers &B, const double *xpos, const uint32_t *gid, cudaStream_t st)
{
    const int L = nlist_lanes(B.n);
    int nb = (int)(((long long)B.n * L + kBlock - 1) / kBlock);
    // in a graph that may skip the pass (the per-step form choice), one wave of
    // blocks striding over the tiles, so that a skipped launch costs little
    if (B.form_sel) nb = std::min(nb, kPassWaveBlocksPerSm * std::max(B.nsm, 1));
    if (L == 1) DTSPH_DISPATCH(B.dim, B.fp32c, (k_pair_cache<D, F32, 1><<<nb, kBlock, 0, st>>>(B, xpos, gid)));
    else if (L == 2) DTSPH_DISPATCH(B.dim, B.fp32c, (k_pair_cache<D, F32, 2><<<nb, kBlock, 0, st>>>(B, xpos, gid)));
    else if (L == 4) DTSPH_DISPATCH(B.dim, B.fp32c, (k_pair_cache<D, F32, 4><<<nb, kBlock, 0, st>>>(B, xpos, gid)));
    else DTSPH_DISPATCH(B.dim, B.fp32c, (k_pair_cache<D, F32, 8><<<nb, kBlock, 0, st>>>(B, xpos, gid)));
    return 1;
}

int launch_shift(const Buffers &B, cudaStream_t st)
{
    const int k = launch_bin_a_to_b(B, st);                   // cells at r^{n+1}
    launch_nlist(B, B.x_b, st);
    DTSPH_DISPATCH(B.dim, B.fp32c, (k_shift<D, F32><<<(B.n + kBlock - 1) / kBlock, kBlock, 0, st>>>(B)));
    return k + 2;
}

}  // namespace dtsph
