// The pseudo-time loop with the particles moving in pseudo-time (Algorithm 1,
// Sec. 2.1 and the "moving" SPH forms of Sec. 3).
//
// One iteration k for every fluid particle (Jacobi, ping-pong on k's parity),
// with the positions carried as r-hat^k = r^{k+1/2} and the pressure as
// p-hat^k = p^{k+1/2}:
//   wall values at the moved fluid positions                       Sec. 3.2
//   rates at (r^{k+1/2}, V^k, p^{k+1/2}, V~^k):
//     dp/dtau = frozen terms + V~_i . sum_j m (p_i + p_j)/rho0^2 gradW_ij    Eq. (dp-dtau)
//     F       = frozen terms + sum_j m/rho0 (V_i + V_j) (V~_i . gradW_ij)   Eq. (discrete_ME)
//   dV/dtau = kappa (F - (3 V^k - 4 V^n + V^{n-1}) / (2 dt))      Eq. (dv_dtau_exact)
//   V^{k+1} = V^k + dtau dV/dtau                                   Eq. (vkp1)
//   V~^{k+1} = dt dV/dtau                                          Eq. (vtilde)
//   r^{k+1} = r^{k+1/2} + dtau/2 V~^{k+1}                          Eq. (rkp1)
//   r^{k+3/2} = r^{k+1} + dtau/2 V~^{k+1}                          Eq. (rkstar), next pass
//   p-hat^{k+1} = p-hat^k + dtau dp/dtau                           Eqs. (pkstar, pkp1)
// The walls stay where they are. The pair geometry changes every pass, so there
// is no pair cache: each pass walks the lists built at r^0 and recomputes r_ij,
// W and gradW from the current positions. With moving = 1 the lists are those
// of r^0 (neighbours not updated); with moving = 2 they are built with the
// cutoff 3h + skin, and a particle that moves farther than skin / 2 from r^0
// raises kErrSkin, so every pair within 3h of the moved positions is listed:
// the sums equal those over neighbours updated at every pass (the pairs beyond
// 3h add exact zeros).
#include <algorithm>

#include "grid_barrier.cuh"
#include "loop_rules.cuh"
#include "pair32.cuh"
#include "pair64.cuh"

namespace dtsph {

namespace {

inline int blocks(int n) { return (n + kBlock - 1) / kBlock; }

// r^{1/2} = r^0 (V~^0 = 0) in both position buffers, V~ = 0. Walls keep r^0 in both buffers for the whole loop.
template <bool F32>
__global__ void __launch_bounds__(kBlock) k_move_init(Buffers B)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B.n || B.gid_a[s] == kNoParticle) return;
    for (int a = 0; a < B.dim; ++a) {
        const size_t q = (size_t)a * B.n + s;
        const double x0 = B.xp_a[q];
        B.xk[0][q] = x0;
        B.xk[1][q] = x0;
        B.vt[q] = 0.0;
    }
    if (F32) {
        B.offk[0][s] = B.off[s];
        B.offk[1][s] = B.off[s];
    }
}

// r_ij = r_i - r_j at the current positions of slots i and j (list entry code
// for the FP32C cell shift), in the working precision; returns |r_ij|^2.
template <int D, bool F32, typename T>
__device__ __forceinline__ T moved_sep(const Geom &G, const Buffers &B, int cur, const T *xi, float4 oi, int j,
                                       int code, T *d)
{
    if (F32) {
        int dx, dy, dz;
        decode_shift(code, dx, dy, dz);
        float f0, f1, f2;
        const float q2 = sep32<D>(shifted_offset<D>(oi, dx, dy, dz, G.s_f), B.offk[cur][j], f0, f1, f2);
        d[0] = (T)f0;
        d[1] = (T)f1;
        if (D == 3) d[2] = (T)f2;
        return (T)q2;
    } else {
        const double *xk = B.xk[cur];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            double v = __dsub_rn((double)xi[a], xk[(size_t)a * B.n + j]);
            if (G.periodic[a]) {
                if (v > G.halfL[a]) v = __dsub_rn(v, G.L[a]);
                else if (v < -G.halfL[a]) v = __dadd_rn(v, G.L[a]);
            }
            d[a] = (T)v;
        }
        T r2 = Ar<T>::add(Ar<T>::mul(d[0], d[0]), Ar<T>::mul(d[1], d[1]));
        if (D == 3) r2 = Ar<T>::add(r2, Ar<T>::mul(d[2], d[2]));
        return r2;
    }
}

// Wall values of iteration k (iterate in buffer cur) at the moved fluid
// positions: p_w = (sum_f p_f W + rho0 g . sum_f r_wf W) / sum_f W and ghost
// velocity 2 v_w - sum_f V_f W / sum_f W (Adami et al., Sec. 3.2), zero when no
// fluid is in range; kept >= 0 in free-surface runs.
template <int D, bool F32>
__device__ __forceinline__ void move_wall(const Buffers &B, const Geom &G, const Phys &P, int cur, int s)
{
    using T = typename std::conditional<F32, float, double>::type;
    T xi[3] = {T(0), T(0), T(0)};
    float4 oi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (F32) {
        oi = B.offk[cur][s];
    } else {
#pragma unroll
        for (int a = 0; a < D; ++a) xi[a] = (T)B.xk[cur][(size_t)a * B.n + s];
    }
    const auto *nb = nb_ptr<T>(B, cur);
    const double sigma = P.sig_h * P.h;
    double sw = 0, sp = 0, sg = 0, sv[3] = {0, 0, 0};
    const uint32_t *lst = slot_list(B, s);
    const int cnt = B.pcount[s];
    for (int k = 0; k < cnt; ++k) {
        const uint32_t jb = lst[k];
        if (jb & kWallBit) continue;            // fluid neighbours only
        const int j = entry_slot(jb);
        T d[3];
        const T r2 = moved_sep<D, F32, T>(G, B, cur, xi, oi, j, entry_code(jb), d);
        const double W = sigma * (double)quintic_w<T>(Ar<T>::mul(sqrt(r2), (T)P.inv_h));
        if (W == 0.0) continue;
        const auto q = nb[j];
        double gr = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) gr += P.g[a] * (double)d[a];
        sw += W;
        sp += (double)q.w * W;
        sg += P.rho0 * gr * W;
        sv[0] += (double)q.x * W;
        sv[1] += (double)q.y * W;
        sv[2] += (double)q.z * W;
    }
    double gv[3];
    for (int a = 0; a < 3; ++a) {
        const double vw = a < D ? B.vn_a[(size_t)a * B.n + s] : 0.0;
        gv[a] = 2.0 * vw - (sw > 0 ? sv[a] / sw : 0.0);
    }
    double pw = sw > 0 ? (sp + sg) / sw : 0.0;
    if (pw < 0.0 && P.free_surface) pw = 0.0;   // free-surface runs (Sec. 3.2)
    if (F32) B.nb32[cur][s] = make_float4((float)gv[0], (float)gv[1], (float)gv[2], (float)pw);
    else B.nb64[cur][s] = make_double4_32a(gv[0], gv[1], gv[2], pw);
}

// One launch per iteration: a thread per slot, wall slots work.
template <int D, bool F32>
__global__ void __launch_bounds__(kBlock) k_move_walls(Buffers B)
{
    __shared__ Geom G;
    __shared__ Phys P;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int inst = block_instance(B, blockIdx.x * kBlock);
    const LoopState *ls = B.ls + inst;
    if (ls->done) return;                       // uniform over the block
    block_copy(G, B.geo[inst]);
    block_copy(P, B.phys[inst]);
    if (s >= B.n) return;
    const uint32_t g = B.gid_a[s];
    if (g < (uint32_t)B.nf || g == kNoParticle) return;
    move_wall<D, F32>(B, G, P, ls->iter & 1, s);
}

// One moving iteration of tile `tile` (kBlock / L slots of instance inst), by the
// whole block: L lanes per slot (lane l takes the list entries, FP32C: pairs of
// entries, l, l + L, ...; the partial sums merge by warp shuffles), then a thread
// per slot for the update. The tile's residual sums come back on thread 0. The pair
// arithmetic is that of the frozen passes (pair32.cuh, pair64.cuh).
template <int D, bool F32, bool WALLS, int L>
__device__ __forceinline__ void move_tile(const Buffers &B, const Geom &G, const Phys &P, const ShiftTable &sh,
                                          double (&red)[2][kBlock / kWarp], int inst, int cur, int tile, double &blk_a,
                                          double &blk_b)
{
    constexpr int PPB = kBlock / L;
    using T = typename std::conditional<F32, float, double>::type;
    __shared__ T part[L > 1 ? 2 * D + 1 : 1][L > 1 ? PPB : 1];
    const int n = B.n, nxt = cur ^ 1;
    int s = tile * PPB + threadIdx.x / L;
    const int lane_in = threadIdx.x % L;
    bool fl = s < n && B.gid_a[s] < (uint32_t)B.nf;
    double r_ap = 0.0, r_av = 0.0;
    // the frozen rates and sum m (p_i + p_j) / rho0^2 gradW_ij
    T apT = T(0), FT[3] = {T(0), T(0), T(0)}, gpT[3] = {T(0), T(0), T(0)};
    const int cnt = fl ? B.pcount[s] : 0;
    const uint32_t *lst = slot_list(B, s);
    if constexpr (F32) {
        const PairK32 k = P.k32;
        const float4 *nb = B.nb32[cur];
        const float4 qi = fl ? nb[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 oi = fl ? B.offk[cur][s] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float vi[3] = {qi.x, qi.y, qi.z};
        Sums32<D> A;
        Move32<D> mv;
#pragma unroll
        for (int a = 0; a < 3; ++a) mv.t[a] = fl && a < D ? (float)B.vt[(size_t)a * n + s] : 0.f;
        auto wall = [&](uint32_t e, const float4 &q, float *w) {
            w[0] = q.x; w[1] = q.y; w[2] = q.z;
            if (e & kWallBit) {
                const float4 v = B.wv32[entry_slot(e)];
                w[0] = v.x; w[1] = v.y; w[2] = v.z;
            }
        };
        list_sums32<D, WALLS, L>(k, sh, lst, cnt, lane_in, oi, vi, qi.w, B.offk[cur], nb, wall, A, mv);
        rates32<D, L>(k, A, apT, FT);
#pragma unroll
        for (int a = 0; a < D; ++a) gpT[a] = -__fmul_rn(k.s_F, merged32<L>(mv.np[a]));
    } else {
        const PairConst<double> k = pair_const<double>(P);
        const double4_32a *nb = B.nb64[cur];
        const double *xk = B.xk[cur];
        const double4_32a qi = fl ? nb[s] : make_double4_32a(0, 0, 0, 0);
        const double vi[3] = {qi.x, qi.y, qi.z};
        double xi[3] = {0, 0, 0}, ti[3] = {0, 0, 0}, gp[3] = {0, 0, 0}, fc[3] = {0, 0, 0};
        if (fl)
            for (int a = 0; a < D; ++a) {
                xi[a] = xk[(size_t)a * n + s];
                ti[a] = B.vt[(size_t)a * n + s];
            }
        Sums64<D> A;
        // R entries per round: their indices, then their gathers, then the pair
        // terms (the entries stay in the order lane_in, lane_in + L, ...)
        constexpr int R = 2;
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
                const double r2 = listed_sep64<D>(G, xi, xk, n, j, d);
                grad64<D>(P, d, r2, g, F);
                const double vv[3] = {qv[r].x, qv[r].y, qv[r].z};
                double vd[3] = {vv[0], vv[1], vv[2]};
                if (WALLS && (jbv[r] & kWallBit)) {
#pragma unroll
                    for (int a = 0; a < D; ++a) vd[a] = B.vn_a[(size_t)a * n + j];
                }
                pair64_accumulate<D, WALLS>(k, g, F, vi, qi.w, vd, vv, qv[r].w, A);
                // advective terms of Eqs. (dp-dtau) and (discrete_ME)
                double tg = 0.0;
#pragma unroll
                for (int a = 0; a < D; ++a) tg = __fma_rn(ti[a], g[a], tg);
                const double pp = __dadd_rn(qi.w, qv[r].w);
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    gp[a] = __fma_rn(pp, g[a], gp[a]);
                    fc[a] = __fma_rn(__dadd_rn(vi[a], vd[a]), tg, fc[a]);
                }
            }
        }
        rates64<D, L>(P, k, A, apT, FT);
#pragma unroll
        for (int a = 0; a < D; ++a) {
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) {
                gp[a] = __dadd_rn(gp[a], __shfl_xor_sync(0xffffffffu, gp[a], o));
                fc[a] = __dadd_rn(fc[a], __shfl_xor_sync(0xffffffffu, fc[a], o));
            }
            gpT[a] = __dmul_rn(__dmul_rn(k.c_p, P.sig_h), gp[a]);
            FT[a] = __fma_rn(__dmul_rn(k.vol, P.sig_h), fc[a], FT[a]);
        }
    }
    // the update: a thread a slot, whole warps (FP64: with the first of a slot's L
    // lanes at work, every FP64 instruction would be issued L times as often)
    if constexpr (L > 1) {
        if (lane_in == 0) {
            const int at = threadIdx.x / L;
            part[0][at] = apT;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                part[1 + a][at] = FT[a];
                part[1 + D + a][at] = gpT[a];
            }
        }
        __syncthreads();
        s = tile * PPB + threadIdx.x;
        fl = threadIdx.x < PPB && s < n && B.gid_a[s] < (uint32_t)B.nf;
        if (threadIdx.x < PPB) {
            apT = part[0][threadIdx.x];
#pragma unroll
            for (int a = 0; a < D; ++a) {
                FT[a] = part[1 + a][threadIdx.x];
                gpT[a] = part[1 + D + a][threadIdx.x];
            }
        }
    }
    if (fl) {
        double xh[3] = {0, 0, 0}, vt[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const size_t q = (size_t)a * n + s;
            xh[a] = B.xk[cur][q];
            vt[a] = B.vt[q];
        }
        // update in FP64
        double apv = (double)apT;
#pragma unroll
        for (int a = 0; a < D; ++a) apv = __fma_rn(vt[a], (double)gpT[a], apv);
        double vnew[3] = {0, 0, 0}, xn[3] = {0, 0, 0};
        double av2 = 0.0;
        const double hdt = 0.5 * P.dtau;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const size_t q = (size_t)a * n + s;
            const double vk = B.vk[cur][q];
            const double Fv = (double)FT[a];
            const double av = __fma_rn(P.kappa, Fv, -__fma_rn(P.kc3, vk, B.s_a[q]));
            vnew[a] = __fma_rn(P.dtau, av, vk);
            B.vk[nxt][q] = vnew[a];
            const double vtn = __dmul_rn(P.dt, av);
            B.vt[q] = vtn;
            const double x1 = __dadd_rn(xh[a], __dmul_rn(hdt, vtn));
            double x2 = __dadd_rn(x1, __dmul_rn(hdt, vtn));
            if (G.periodic[a]) {
                if (x2 >= G.hi[a]) x2 = __dsub_rn(x2, G.L[a]);
                else if (x2 < G.lo[a]) x2 = __dadd_rn(x2, G.L[a]);
            }
            xn[a] = x2;
            B.xk[nxt][q] = x2;
            av2 = __fma_rn(av, av, av2);
        }
        if (F32) {
            // offsets from the slot's cell origin at r^0 (minimum image)
            const int lc = B.cell_a[s] - B.inst[inst].cell_off;
            const int c[3] = {lc % G.nc[0], (lc / G.nc[0]) % G.nc[1], lc / (G.nc[0] * G.nc[1])};
            float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int a = 0; a < D; ++a) {
                double v = xn[a] - (G.lo[a] + c[a] * G.s[a]);
                if (G.periodic[a]) {
                    if (v > G.halfL[a]) v -= G.L[a];
                    else if (v < -G.halfL[a]) v += G.L[a];
                }
                o[a] = (float)v;
            }
            B.offk[nxt][s] = make_float4(o[0], o[1], o[2], 0.f);
            const float pnew = __fmaf_rn(P.dtau_f, (float)apv, B.nb32[cur][s].w);
            B.nb32[nxt][s] = make_float4((float)vnew[0], (float)vnew[1], (float)vnew[2], pnew);
        } else {
            const double pnew = __fma_rn(P.dtau, apv, B.nb64[cur][s].w);
            B.nb64[nxt][s] = make_double4_32a(vnew[0], vnew[1], vnew[2], pnew);
        }
        if (P.moving == 2) {
            // the lists cover displacements up to skin / 2 from r^0
            double d2 = 0.0;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                double v = xn[a] - B.xp_a[(size_t)a * n + s];
                if (G.periodic[a]) {
                    if (v > G.halfL[a]) v -= G.L[a];
                    else if (v < -G.halfL[a]) v += G.L[a];
                }
                d2 += v * v;
            }
            if (!(d2 < P.disp2_max)) atomicOr(B.err, kErrSkin);
        }
        r_ap = fabs(apv);
        r_av = sqrt(av2);
    }
    // fixed-order block sum of the residual terms
    const double w_ap = warp_sum<double>(r_ap), w_av = warp_sum<double>(r_av);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = w_ap;
        red[1][threadIdx.x >> 5] = w_av;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        blk_a = blk_b = 0;
        for (int w = 0; w < kBlock / kWarp; ++w) {
            blk_a += red[0][w];
            blk_b += red[1][w];
        }
    }
    __syncthreads();   // red is reused
}

// One launch per iteration: one tile per block; the last block of an instance
// applies its stop rules, the last block of all sets the while-node condition (as
// the frozen iterate kernel).
template <int D, bool F32, bool WALLS, int L>
__global__ void __launch_bounds__(kBlock) k_move_iter(Buffers B, unsigned long long cond, int use_cond)
{
    constexpr int PPB = kBlock / L;
    __shared__ Geom G;
    __shared__ Phys P;
    __shared__ ShiftTable sh;
    __shared__ double red[2][kBlock / kWarp];
    __shared__ int last, tlo_sh;
    if (!use_cond && B.ctrl->active == 0) return;   // whole grid agrees: nothing to do
    const int inst = block_instance(B, blockIdx.x * PPB);
    LoopState *ls = B.ls + inst;
    int tlo, thi;
    instance_tiles(B.inst[inst], PPB, tlo, thi);
    const bool mine = (int)blockIdx.x < thi;        // false: a tile made of padding only
    const int it = ls->iter;
    const bool work = mine && !ls->done;
    if (work) {
        if (F32) load_shifts(sh, B.geo[inst]);
        block_copy(G, B.geo[inst]);
        block_copy(P, B.phys[inst]);
        double a, b;
        move_tile<D, F32, WALLS, L>(B, G, P, sh, red, inst, it & 1, blockIdx.x, a, b);
        if (threadIdx.x == 0) {
            B.blk[2 * blockIdx.x] = a;
            B.blk[2 * blockIdx.x + 1] = b;
            __threadfence();
            const unsigned int t = atomicAdd(&ls->ticket, 1u);
            last = (t == (unsigned int)(thi - tlo - 1));
            tlo_sh = tlo;
        }
        __syncthreads();
        if (last) {
            // last tile of this instance: fixed-order reduction of its partials
            __threadfence();
            double sa = 0, sb = 0;
            reduce_tiles(B.blk + 2 * tlo_sh, thi - tlo_sh, red, sa, sb);
            if (threadIdx.x == 0) {
                const int r = finish_iteration(ls, P, it, sa, sb);
                ls->ticket = 0;
                if (r != -1) atomicSub(&B.ctrl->active, 1);
                __threadfence();
            }
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int t = atomicAdd(&B.ctrl->ticket, 1u);
        if (t == gridDim.x - 1) {
            B.ctrl->ticket = 0;
            __threadfence();
            const int active = *(volatile int *)&B.ctrl->active;
            if (use_cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond, active > 0 ? 1u : 0u);
        }
    }
}

// Every moving iteration of one real step of one instance in one cooperative launch
// (as k_loop for particles fixed in pseudo-time; the same tiles, sums and
// decisions as k_move_iter). A small problem's pass is bound by the latency of its
// gathers and the while node adds two launches and a last-block reduction to each:
// iteration of 151 x 151 particles, FP32C, 24 -> 16.8 us. Batches keep the while
// node: their instances stop at different iterations.
template <int D, bool F32, bool WALLS, int L>
__global__ void __launch_bounds__(kBlock, F32 ? 2 : 1) k_move_loop(Buffers B)
{
    constexpr int PPB = kBlock / L;
    __shared__ LoopState st;
    __shared__ Geom G;
    __shared__ Phys P;
    __shared__ ShiftTable sh;
    __shared__ double red[2][kBlock / kWarp];
    __shared__ int stop, ok_sh;
    if (threadIdx.x == 0) {
        st = *B.ls;
        stop = 0;
    }
    if (F32) load_shifts(sh, B.geo[0]);
    block_copy(G, B.geo[0]);
    block_copy(P, B.phys[0]);                       // (ends with a barrier)
    int tlo, ntiles;
    instance_tiles(B.inst[0], PPB, tlo, ntiles);    // (one instance: from slot 0)
    unsigned int epoch = 0;
    int r = -1, it = st.iter;
    for (;; ++it) {
        const int cur = it & 1;
        if constexpr (WALLS) {
            // the wall list's warps dealt to the blocks in turn (eight to a block, the FP64
            // sums of 3,000 walls kept 12 SMs busy and the others waiting: two steps of a 250 x
            // 250 FP32C cavity 4.1 ms, so 2.2)
            for (int w = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * kWarp + (threadIdx.x & 31); w < B.nw;
                 w += (kBlock / kWarp) * gridDim.x * kWarp)
                move_wall<D, F32>(B, G, P, cur, B.wslot_a[w]);
            if (!grid_barrier<false>(&B.ctrl->bar, ++epoch, B.err, ok_sh, B.barrier_ns)) break;
        }
        double *blk = B.blk + (size_t)cur * 2 * ntiles;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            double a, b;
            move_tile<D, F32, WALLS, L>(B, G, P, sh, red, 0, cur, t, a, b);
            if (threadIdx.x == 0) {
                blk[2 * t] = a;
                blk[2 * t + 1] = b;
            }
        }
        if (!grid_barrier<false>(&B.ctrl->bar, ++epoch, B.err, ok_sh, B.barrier_ns)) break;
        double sa = 0, sb = 0;
        reduce_tiles(blk, ntiles, red, sa, sb);
        if (threadIdx.x == 0) {
            st.rp = sa * P.rp_scale;
            st.rv = sb * P.rv_scale;
            st.hist_p[it & 15] = st.rp;
            st.hist_v[it & 15] = st.rv;
            r = stop_rule(st, it + 1);
            stop = r != -1;
        }
        __syncthreads();
        if (stop) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        LoopState *ls = B.ls;
        ls->rp = st.rp;
        ls->rv = st.rv;
        for (int q = 0; q < 16; ++q) {
            ls->hist_p[q] = st.hist_p[q];
            ls->hist_v[q] = st.hist_v[q];
        }
        ls->iter = stop ? it + 1 : it;
        ls->reason = stop ? r : 3;                  // (a barrier that gave up: the step is reported)
        ls->done = 1;
    }
}

template <int D, bool F32, bool WALLS>
const void *move_loop_lanes(int lanes)
{
    switch (lanes) {
    case 1: return (const void *)k_move_loop<D, F32, WALLS, 1>;
    case 2: return (const void *)k_move_loop<D, F32, WALLS, 2>;
    case 4: return (const void *)k_move_loop<D, F32, WALLS, 4>;
    default: return (const void *)k_move_loop<D, F32, WALLS, 8>;
    }
}

}  // namespace

const void *move_loop_function(const Buffers &B)
{
    const void *fn = nullptr;
    DTSPH_DISPATCH(B.dim, B.fp32c, {
        fn = B.nw > 0 ? move_loop_lanes<D, F32, true>(B.lanes) : move_loop_lanes<D, F32, false>(B.lanes);
    });
    return fn;
}

int launch_move_prepare(const Buffers &B, cudaStream_t st)
{
    launch_nlist(B, B.xp_a, st);
    if (B.fp32c) k_move_init<true><<<blocks(B.n), kBlock, 0, st>>>(B);
    else k_move_init<false><<<blocks(B.n), kBlock, 0, st>>>(B);
    return 2;
}

int launch_move_iteration(const Buffers &B, unsigned long long cond, int use_cond, cudaStream_t st)
{
    int k = 0;
    if (B.nw > 0) {
        DTSPH_DISPATCH(B.dim, B.fp32c, (k_move_walls<D, F32><<<blocks(B.n), kBlock, 0, st>>>(B)));
        ++k;
    }
    // n is a multiple of kSlotAlign, so the tiles of kBlock / L slots cover it exactly
    const int L = B.lanes, nb = (int)((long long)B.n * L / kBlock);
    auto go = [&](auto lanes) {
        constexpr int LL = decltype(lanes)::value;
        if (B.nw > 0) DTSPH_DISPATCH(B.dim, B.fp32c, (k_move_iter<D, F32, true, LL><<<nb, kBlock, 0, st>>>(B, cond, use_cond)));
        else DTSPH_DISPATCH(B.dim, B.fp32c, (k_move_iter<D, F32, false, LL><<<nb, kBlock, 0, st>>>(B, cond, use_cond)));
    };
    switch (L) {
    case 1: go(std::integral_constant<int, 1>()); break;
    case 2: go(std::integral_constant<int, 2>()); break;
    case 4: go(std::integral_constant<int, 4>()); break;
    default: go(std::integral_constant<int, 8>()); break;
    }
    return k + 1;
}

}  // namespace dtsph
