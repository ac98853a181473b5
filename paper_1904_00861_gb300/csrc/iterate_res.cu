// The resident pseudo-time loop: the persistent loop of one instance whose
// particles fit one block per SM (FP32C up to 87,552 slots, FP64 48,640, at one lane
// each on 152 SMs).
//
// On such sizes k_loop's iteration is a chain of latencies, not of bytes: cache
// rows from L2, then the neighbour gathers, a few entries at a time; loads and
// stores of the velocity iterate; then the grid barrier, the reduction of the
// residual partials and the stop rules, with nothing else running. Here every block
// keeps its slots for the whole step:
//  - their cache rows are copied to shared memory once (as many as fit; the rest
//    are read from L2 as before), so a lane's gathers go out at once, eight in
//    flight;
//  - V^k, p-hat and the BDF2 source stay in registers, and only the packed (V,
//    p-hat) that neighbours gather is written each iteration;
//  - two warps more per block reduce the residual partials of the iteration before
//    and apply the stop rules while the others run the next pair sums (which
//    write nothing until that decision is in).
// An iteration, k_loop -> here: 200 x 200 FP32C 14.0 -> 9.6 us (cycles: pair sums
// and decision side by side 9,500, update 4,500, barrier 3,000), FP64 60 -> 37 us
// (the FP64 pipe); 50 x 50 FP64 14.4 -> 9.4 us; cavity 200 x 200 with 2,436 walls
// 32 -> 15 us; dam break of 20,402 particles 26 -> 12.6 us.
// Every sum is formed in the order of k_iterate at the same lanes: pairs by lane,
// residuals by warps of 32 slots, tiles of 256 / L slots, and reduce_tiles' order,
// so the bits are those of the other drivers.
#include <algorithm>
#include <type_traits>

#include "loop_kernels.cuh"

namespace dtsph {

namespace {

constexpr int kDecide = 64;                   // threads that reduce the residuals and decide
// Most threads that work on slots (L a slot): with those that decide, 640 leave 96
// registers a thread, 384 leave 168.
template <bool F32>
constexpr int kResThreads = F32 ? 576 : 320;
constexpr int kResTiles = 384;                // most residual tiles of such an instance

// Cache rows of a block in shared memory: row r of thread t at r W + t in each array.
template <bool F32> struct ResRows;
template <> struct ResRows<true> {
    float4 *c0, *c1;
    uint2 *e;           // 3D
};
template <> struct ResRows<false> {
    double2 *c0, *c1;
    uint32_t *e;
};

template <int D, bool F32>
__host__ __device__ constexpr int row_bytes() { return F32 ? (D == 2 ? 32 : 40) : 36; }

// Tile sums of an iteration by `threads` threads (thread `at` of them): tile t is
// the groups (32 slots) t G .. t G + G - 1 added in order.
template <int G>
__device__ __forceinline__ void tile_sums(const double *blk, int ntiles, double2 *tile, int at, int threads)
{
    const double2 *g = reinterpret_cast<const double2 *>(blk);
#pragma unroll 4
    for (int t = at; t < ntiles; t += threads) {
        double2 v[G];
#pragma unroll
        for (int i = 0; i < G; ++i) v[i] = __ldcg(g + t * G + i);
#pragma unroll
        for (int i = 1; i < G; ++i) {
            v[0].x += v[i].x;
            v[0].y += v[i].y;
        }
        tile[t] = v[0];
    }
}

// The sum of the tiles in reduce_tiles' order (256 strided lanes, butterflies of 32,
// their totals in order) by one warp, both quantities: a on lanes 0-15, b on 16-31.
// The 16 butterflies (8 strided groups, two quantities) run together, each
// step halving the rows a lane carries, so they take 16 additions, not 80.
__device__ __forceinline__ double sum_tiles(const double2 *tile, int ntiles)
{
    static_assert(kResTiles <= 512, "two strided terms");
    const int lane = threadIdx.x & 31;
    double x[16];
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int t = w * 32 + lane;
        double2 v = t < ntiles ? tile[t] : make_double2(0.0, 0.0);
        if (t + 256 < ntiles) {
            const double2 u = tile[t + 256];
            v.x += u.x;
            v.y += u.y;
        }
        x[w] = v.x;
        x[8 + w] = v.y;
    }
#pragma unroll
    for (int o = 16, rows = 8; o > 1; o >>= 1, rows >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < rows; ++i) {
            const double keep = up ? x[i + rows] : x[i], give = up ? x[i] : x[i + rows];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    const double v = x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
    // lane bits 3, 2, 1 are the group's bits 2, 1, 0
    double sum = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) sum += __shfl_sync(0xffffffffu, v, (lane & 16) | w << 1);
    return sum;
}

template <int D, bool F32, bool WALLS, int L>
__global__ void __launch_bounds__(kResThreads<F32> + kDecide, 1) k_loop_res(Buffers B)
{
    using T = Real<F32>;
    __shared__ LoopState st;
    __shared__ Phys P;
    __shared__ int stop, why, ok_sh;
    __shared__ double2 tile[kResTiles];
    if constexpr (!WALLS) {
        if (skip_form(B)) return;         // the step runs the other pair-term form
    }
    const int Q = B.res_q, W = Q * L, rows = B.res_rows, n = B.n;
    const int tid = threadIdx.x, base = blockIdx.x * Q;
    T *part = reinterpret_cast<T *>(dyn_smem);           // [D + 1][Q] rates between the phases (L > 1)
    unsigned char *rbase = dyn_smem + (L > 1 ? (size_t)(D + 1) * Q * sizeof(T) : 0);
    ResRows<F32> rw;
    rw.c0 = reinterpret_cast<decltype(rw.c0)>(rbase);
    rw.c1 = rw.c0 + (size_t)rows * W;
    rw.e = reinterpret_cast<decltype(rw.e)>(rw.c1 + (size_t)rows * W);
    if (tid == 0) {
        st = *B.ls;
        stop = 0;
        why = -1;
    }
    block_copy(P, B.phys[0]);                            // (ends with a barrier)
    const bool worker = tid < W;
    // phase 1: L threads a slot
    const int s = base + tid / L, lane_in = tid % L;
    const bool active = worker && s < n && B.gid_a[s] < (uint32_t)B.nf;
    const int cnt = active ? B.pcount[s] : 0;
    const int items = F32 ? list_pairs(cnt) : cnt;       // records of the slot, lane l takes l, l + L, ...
    const int nr = items > lane_in ? (items - lane_in + L - 1) / L : 0;
    const size_t row0 = F32 ? cache_row(B, s) : (size_t)(s >> 5) * B.K;
    for (int r = 0; r < min(nr, rows); ++r) {
        const int m = lane_in + r * L, at = r * W + tid;
        if constexpr (F32) {
            const CachePair c = cache_pair<D>(B, row0 + m, s & 31);
            rw.c0[at] = c.c0;
            rw.c1[at] = c.c1;
            if constexpr (D == 3) rw.e[at] = make_uint2(c.ea, c.eb);
        } else {
            const size_t e = (row0 + m) * kWarp + (s & 31);
            const double4_32a c = B.pc64[e];
            rw.c0[at] = make_double2(c.x, c.y);
            rw.c1[at] = make_double2(c.z, c.w);
            rw.e[at] = B.pj[e];
        }
    }
    // phase 2: one thread a slot
    int it = st.iter;
    const int it0 = it;
    const int s2 = base + tid;
    const bool slot2 = tid < Q && s2 < n;
    const bool fl = slot2 && B.gid_a[s2] < (uint32_t)B.nf;
    double vk[3] = {0, 0, 0}, src[3] = {0, 0, 0};
    T p = T(0);
    if (fl) {
        for (int a = 0; a < D; ++a) {
            vk[a] = B.vk[it & 1][(size_t)a * n + s2];
            src[a] = B.s_a[(size_t)a * n + s2];
        }
        if constexpr (F32) p = B.nb32[it & 1][s2].w;
        else p = B.nb64[it & 1][s2].w;
    }
    constexpr int PPB = kBlock / L, G = PPB / kWarp;
    const int ngroups = n / kWarp;
    // iteration it - 1's residuals and the stop rules, by the last two warps
    auto decide = [&](int it) {
        if (it == it0) return;                           // nothing done yet in this launch
        int tlo, thi;
        instance_tiles(B.inst[0], PPB, tlo, thi);
        tile_sums<G>(B.blk + (size_t)((it - 1) & 1) * 2 * ngroups, thi, tile, tid - W, kDecide);
        asm volatile("bar.sync 1, %0;" ::"n"(kDecide) : "memory");
        if (tid >= W + kWarp) return;
        const double sa = sum_tiles(tile, thi);
        const double sb = __shfl_sync(0xffffffffu, sa, 16);
        if (tid == W) {
            st.rp = sa * P.rp_scale;
            st.rv = sb * P.rv_scale;
            st.hist_p[(it - 1) & 15] = st.rp;
            st.hist_v[(it - 1) & 15] = st.rv;
            why = stop_or_pause(st, it);
            stop = why != -1;
        }
    };
    unsigned int epoch = 0;
    for (;; ++it) {
        const int cur = it & 1;
        if constexpr (WALLS) {
            // the wall list, kWallLanes threads per wall particle, its warps dealt to the
            // blocks in turn
            if (worker) {
                int sub;
                unsigned gmask;
                wall_group(tid, sub, gmask);
                constexpr int WPW = kWarp / kWallLanes;
                for (int w = ((tid >> 5) * gridDim.x + blockIdx.x) * WPW + (tid & 31) / kWallLanes; w < B.nw;
                     w += (W >> 5) * gridDim.x * WPW)
                    wall_slot<D, F32>(B, B.wslot_a[w], cur, sub, gmask);
            } else {
                decide(it);
            }
            __syncthreads();
            if (stop) break;
            if (!grid_barrier<true>(&B.ctrl->bar, ++epoch, B.err, ok_sh, B.barrier_ns)) break;
        }
        T apT = T(0), FT[3] = {T(0), T(0), T(0)};
        if (worker) {
            if constexpr (F32) {
                const PairK32 k = P.k32;
                const float4 *nb = B.nb32[cur];
                const float4 qi = active ? nb[s] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float vi[3] = {qi.x, qi.y, qi.z};
                Sums32<D> A;
                NoMove mv;
                // the terms of records r0 .. r0 + R - 1 (those below nr), the gathers together
                auto terms = [&](auto in_smem, int r0) {
                    constexpr int R = decltype(in_smem)::value ? 4 : 2;
                    uint32_t e[2 * R];
                    float4 q[2 * R];
                    float w[2 * R][3];
                    CachePair c[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int r = min(r0 + i, nr - 1);
                        uint2 v;
                        if constexpr (decltype(in_smem)::value) {
                            const int at = min(r, rows - 1) * W + tid;
                            v = D == 3 ? rw.e[at] : reinterpret_cast<const uint2 *>(rw.c1 + at)[1];
                        } else {
                            c[i] = cache_pair<D>(B, row0 + lane_in + (size_t)r * L, s & 31);
                            v = make_uint2(c[i].ea, c[i].eb);
                        }
                        e[2 * i] = v.x;
                        e[2 * i + 1] = v.y;
                    }
#pragma unroll
                    for (int i = 0; i < 2 * R; ++i) {
                        q[i] = nb[WALLS ? e[i] & ~kWallBit : e[i]];
                        if constexpr (WALLS) {
                            w[i][0] = q[i].x; w[i][1] = q[i].y; w[i][2] = q[i].z;
                            if (e[i] & kWallBit) {
                                const float4 v = B.wv32[e[i] & ~kWallBit];
                                w[i][0] = v.x; w[i][1] = v.y; w[i][2] = v.z;
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int r = r0 + i;
                        if (r >= (decltype(in_smem)::value ? min(nr, rows) : nr)) break;
                        if constexpr (decltype(in_smem)::value) {
                            c[i].c0 = rw.c0[r * W + tid];
                            c[i].c1 = rw.c1[r * W + tid];
                        }
                        F2 g[D], F;
                        cache_coefs<D>(c[i], g, F);
                        pair2_accumulate<D, WALLS>(k, g, F, vi, qi.w, q[2 * i], q[2 * i + 1], w[2 * i], w[2 * i + 1], A,
                                                   mv);
                    }
                };
                for (int r0 = 0; r0 < min(nr, rows); r0 += 4) terms(std::true_type(), r0);
                for (int r0 = rows; r0 < nr; r0 += 2) terms(std::false_type(), r0);
                rates32<D, L>(k, A, apT, FT);
            } else {
                const PairConst<double> k = pair_const<double>(P);
                const double4_32a *nb = B.nb64[cur];
                const double4_32a qi = active ? nb[s] : make_double4_32a(0, 0, 0, 0);
                const double vi[3] = {qi.x, qi.y, qi.z};
                Sums64<D> A;
                constexpr int R = 4;
                for (int r0 = 0; r0 < nr; r0 += R) {
                    uint32_t e[R];
                    double4_32a c[R], q[R];
                    double w[R][3];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int r = min(r0 + i, nr - 1), at = r * W + tid;
                        if (r < rows) {
                            const double2 x = rw.c0[at], y = rw.c1[at];
                            c[i] = make_double4_32a(x.x, x.y, y.x, y.y);
                            e[i] = rw.e[at];
                        } else {
                            const size_t f = (row0 + lane_in + (size_t)r * L) * kWarp + (s & 31);
                            c[i] = B.pc64[f];
                            e[i] = B.pj[f];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        q[i] = nb[e[i] & ~kWallBit];
                        if constexpr (WALLS) wall_velocity<D>(B, e[i], w[i]);
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if (r0 + i >= nr) break;
                        const double g[3] = {c[i].x, c[i].y, c[i].z};
                        const double vj[3] = {q[i].x, q[i].y, q[i].z};
                        if constexpr (WALLS) {
                            const bool wall = (e[i] & kWallBit) != 0;
                            const double vd[3] = {wall ? w[i][0] : vj[0], wall ? w[i][1] : vj[1], wall ? w[i][2] : vj[2]};
                            pair64_accumulate<D, true>(k, g, c[i].w, vi, qi.w, vd, vj, q[i].w, A);
                        } else {
                            pair64_accumulate<D, false>(k, g, c[i].w, vi, qi.w, vj, vj, q[i].w, A);
                        }
                    }
                }
                rates64<D, L>(P, k, A, apT, FT);
            }
            if constexpr (L > 1) {
                if (lane_in == 0) {
                    part[tid / L] = apT;
#pragma unroll
                    for (int a = 0; a < D; ++a) part[(1 + a) * Q + tid / L] = FT[a];
                }
            }
        } else if constexpr (!WALLS) {
            decide(it);
        }
        __syncthreads();
        if constexpr (!WALLS) {
            if (stop) break;
        }
        if (tid < Q) {
            if constexpr (L > 1) {
                apT = part[tid];
#pragma unroll
                for (int a = 0; a < D; ++a) FT[a] = part[(1 + a) * Q + tid];
            }
            double w_ap, w_av;
            update_slot<D, F32>(P, fl, apT, FT, vk, src, p, w_ap, w_av);
            if (fl) store_state<D, F32>(B, cur ^ 1, s2, vk, p);
            if (slot2 && (tid & 31) == 0) {
                double *g = B.blk + (size_t)cur * 2 * ngroups + 2 * (s2 / kWarp);
                g[0] = w_ap;
                g[1] = w_av;
            }
        }
        if (!grid_barrier<true>(&B.ctrl->bar, ++epoch, B.err, ok_sh, B.barrier_ns)) break;
    }
    // `it` iterations are done (a barrier that gave up: the step is reported)
    if (fl)
        for (int a = 0; a < D; ++a) B.vk[it & 1][(size_t)a * n + s2] = vk[a];
    if (blockIdx.x == 0 && tid == 0) {
        LoopState *ls = B.ls;
        ls->rp = st.rp;
        ls->rv = st.rv;
        for (int q = 0; q < 16; ++q) {
            ls->hist_p[q] = st.hist_p[q];
            ls->hist_v[q] = st.hist_v[q];
        }
        ls->iter = it;
        ls->reason = stop ? why : 3;
        ls->done = 1;
    }
}

template <int D, bool F, bool W>
const void *res_lanes(int lanes)
{
    switch (lanes) {
    case 1: return (const void *)k_loop_res<D, F, W, 1>;
    case 2: return (const void *)k_loop_res<D, F, W, 2>;
    case 4: return (const void *)k_loop_res<D, F, W, 4>;
    default: return (const void *)k_loop_res<D, F, W, 8>;
    }
}

template <bool W>
const void *res_function(const Buffers &B)
{
    if (B.dim == 2) return B.fp32c ? res_lanes<2, true, W>(B.lanes) : res_lanes<2, false, W>(B.lanes);
    return B.fp32c ? res_lanes<3, true, W>(B.lanes) : res_lanes<3, false, W>(B.lanes);
}

// Dynamic shared memory a block may take beside the kernel's own.
constexpr size_t kResSmem = 232448 - 10 * 1024;

}  // namespace

bool resident_shape(const Buffers &B, ResShape *S)
{
    if (B.ninst != 1 || B.form_a || B.xk[0] || B.nsm < 1) return false;
    const int groups = B.n / kWarp;
    const int q = (groups + B.nsm - 1) / B.nsm * kWarp;
    if (q * B.lanes > (B.fp32c ? kResThreads<true> : kResThreads<false>) || B.n / (kBlock / B.lanes) > kResTiles) return false;
    S->q = q;
    S->grid = (B.n + q - 1) / q;
    S->threads = q * B.lanes + kDecide;
    const size_t part = B.lanes > 1 ? (size_t)(B.dim + 1) * q * (B.fp32c ? 4 : 8) : 0;
    const size_t row = (size_t)q * B.lanes * (B.fp32c ? (B.dim == 2 ? row_bytes<2, true>() : row_bytes<3, true>()) : row_bytes<2, false>());
    const int most = ((B.fp32c ? cache_rows(B.K) : B.K) + B.lanes - 1) / B.lanes;
    S->rows = (int)std::min<size_t>(most, (kResSmem - part) / row);
    S->smem = part + (size_t)S->rows * row;
    S->fn = B.nw > 0 ? res_function<true>(B) : res_function<false>(B);
    return true;
}

int resident_prepare()
{
    Buffers B = {};
    for (int dim = 2; dim <= 3; ++dim)
        for (int f = 0; f < 2; ++f)
            for (int lanes = 1; lanes <= 8; lanes *= 2) {
                B.dim = dim;
                B.fp32c = f;
                B.lanes = lanes;
                if (cudaFuncSetAttribute(res_function<true>(B), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kResSmem) != cudaSuccess ||
                    cudaFuncSetAttribute(res_function<false>(B), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kResSmem) != cudaSuccess)
                    return -1;
            }
    return 0;
}

}  // namespace dtsph
