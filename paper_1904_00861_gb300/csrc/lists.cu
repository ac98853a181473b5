// Neighbour lists N(i) = {j != i : |r_ij| < 3h} (Sec. 3; 3h + skin for moving
// particles with neighbour updates, 3h + list_skin for lists reused at the next
// r^n) of every slot, from the cell binning.
//
// Two builders, same lists in the same order:
//  - k_nlist_home: the home particles in the lanes (a row segment of three cells
//    in 2D, a cell in 3D), the candidates broadcast from shared memory;
//  - k_nlist_cells2, small 2D problems: one warp per home cell, the candidates in
//    the lanes. The warp stages the particles of the 9 surrounding cells in shared
//    memory, in the order rows (dy), then dx, then slot, each tagged with its list
//    entry (slot, cell shift code, wall flag); then, for every chunk of 32 staged
//    candidates (one per lane) and every home particle in turn, each lane tests its
//    candidate against that home particle. A ballot ranks the hits, which join the
//    home particle's list as one contiguous run.
// The lists are written per slot (slot s at s Ks + k, Ks = K rounded up to 8), each
// row filled up to a multiple of four with entries of the slot itself, where
// every pass reads them.
//
// The tests are those of the neighbour definition: FP64 positions, squares
// summed in axis order without FMA, minimum image on periodic axes. Both
// precisions first test the FP32 separation from cell offsets and take the FP64
// test only inside a thin band around the cutoff, so both give the same sets, in
// the same order.
#include "f32x2.cuh"
#include "geometry.cuh"

namespace dtsph {

namespace {

constexpr int kWarpsPerBlock = kBlock / kWarp;

// Global row segment g -> its instance (segments of instance i start at inst[i].seg_off).
__device__ __forceinline__ int segment_instance(const Buffers &B, int g)
{
    int lo = 0, hi = B.ninst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.inst[mid].seg_off <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Global cell c -> its instance (cells of instance i start at inst[i].cell_off).
__device__ __forceinline__ int cell_instance(const Buffers &B, int c)
{
    int lo = 0, hi = B.ninst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.inst[mid].cell_off <= c) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// 2D lists of small problems, one warp per cell with the candidates in the lanes
// (see the top of the file).
__global__ void __launch_bounds__(kBlock) k_nlist_cells2(Buffers B, const double *xpos,
                                                         uint32_t *__restrict__ lists, int Ks)
{
    grid_start<false>();
    if (skip_relist(B)) return;   // (the step graph: relisting or not)
    constexpr int NC = 9;                               // surrounding cells
    constexpr int CH = 256;                             // staged candidates per round
    __shared__ float4 cand[kWarpsPerBlock][CH];         // cell offsets, .w = list entry bits
    __shared__ float4 home[kWarpsPerBlock][kWarp];
    __shared__ int tpre[kWarpsPerBlock][NC + 1];        // candidates before surrounding cell t
    __shared__ int tbeg[kWarpsPerBlock][NC];            // first slot of surrounding cell t
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & (kWarp - 1), w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int c = blockIdx.x * kWarpsPerBlock + w;      // global cell of this warp
    if (c >= B.ncell) return;                           // whole warp
    const int inst = cell_instance(B, c);
    const int cell_off = B.inst[inst].cell_off;
    const Geom &G = B.geo[inst];
    const int nx = G.nc[0], ny = G.nc[1];
    const int lc = c - cell_off;
    if (lc >= nx * ny) return;                          // the instance's empty sentinel cell
    const int *start = B.cell_start + cell_off;
    const int hb = start[lc], he = start[lc + 1];
    if (hb == he) return;
    const int cx = lc % nx, cy = lc / nx;
    const float sf[3] = {G.s_f[0], G.s_f[1], 0.f};
    const float rc2_lo = G.rc2_lo, rc2_hi = G.rc2_hi;
    const double rc2 = G.rc2;
    // squared distance from the home cell beyond which no home particle can reach
    // a candidate (the band's top, with a margin far above the rounding of FP32
    // offsets, which lie in [0, s])
    const float box_cut2 = rc2_hi * 1.001f;
    const int n = B.n, K = B.K;
    // the surrounding cells side by side: lane t takes shift code (dx + 1) +
    // 3 (dy + 1) (+ 9: dz = 0); empty when off a closed edge
    int m = 0;
    if (lane < NC) {
        const int dx = lane % 3 - 1, dy = lane / 3 - 1;
        int x = cx + dx, y = cy + dy;
        bool ok = true;
        if (x < 0 || x >= nx) { if (G.periodic[0]) x = x < 0 ? x + nx : x - nx; else ok = false; }
        if (y < 0 || y >= ny) { if (G.periodic[1]) y = y < 0 ? y + ny : y - ny; else ok = false; }
        if (ok) {
            const int nc = y * nx + x;
            const int jb = start[nc];
            m = start[nc + 1] - jb;
            tbeg[w][lane] = jb;
        } else {
            tbeg[w][lane] = 0;
        }
    }
    int incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane < NC) tpre[w][lane] = incl - m;
    const int total = __shfl_sync(full, incl, NC - 1);
    if (lane == NC) tpre[w][NC] = total;
    __syncwarp();
    for (int h0 = hb; h0 < he; h0 += kWarp) {
        const int nh = min(kWarp, he - h0);
        // the home particles of this round, one per lane, into shared memory
        if (lane < nh) home[w][lane] = B.off[h0 + lane];
        int cnt = 0;                                    // list length of home particle h0 + lane
        int t = 0;                                      // surrounding cell of the next fill position
        for (int c0 = 0; c0 < total; c0 += CH) {
            const int span = min(total - c0, CH);
            // fill: stream position p is candidate p - tpre[t] of surrounding
            // cell t; a candidate farther than the cutoff from every point of the
            // home cell (the outer parts of the edge and corner cells) is dropped
            // for the whole warp; the others keep their order
            int take = 0;
            for (int q0 = 0; q0 < span; q0 += kWarp) {
                const int q = q0 + lane;
                bool keep = false;
                float4 e;
                if (q < span) {
                    const int p = c0 + q;
                    while (tpre[w][t + 1] <= p) ++t;
                    const int j = tbeg[w][t] + (p - tpre[w][t]);
                    const int dx = t % 3 - 1, dy = t / 3 - 1;
                    const float4 oj = B.off[j];
                    e = oj;
                    e.w = __uint_as_float(list_entry((uint32_t)j, t + 9, oj.w != 0.f));
                    const float ex = __fadd_rn(oj.x, (float)dx * sf[0]);
                    const float ey = __fadd_rn(oj.y, (float)dy * sf[1]);
                    const float bx = fmaxf(fmaxf(-ex, ex - sf[0]), 0.f);
                    const float by = fmaxf(fmaxf(-ey, ey - sf[1]), 0.f);
                    keep = bx * bx + by * by < box_cut2;
                }
                const unsigned bal = __ballot_sync(full, keep);
                if (keep) cand[w][take + __popc(bal & lt)] = e;
                take += __popc(bal);
            }
            __syncwarp();
            for (int q0 = 0; q0 < take; q0 += kWarp) {
                const bool valid = q0 + lane < take;
                float4 e;
                uint32_t ej = kNoParticle;
                if (valid) {
                    e = cand[w][q0 + lane];
                    ej = __float_as_uint(e.w);
                }
                const int j = entry_slot(ej);
                int dx, dy, dz;
                decode_shift(entry_code(ej), dx, dy, dz);
                for (int h = 0; h < nh; ++h) {
                    const int s = h0 + h;
                    const float4 oi = home[w][h];
                    float f0, f1, f2;
                    const float q2 = sep32<2>(shifted_offset<2>(oi, dx, dy, dz, sf), e, f0, f1, f2);
                    const bool cand_ok = valid && j != s;
                    bool in = cand_ok && q2 < rc2_lo;
                    const bool band = cand_ok && q2 >= rc2_lo && q2 < rc2_hi;
                    // the FP64 decision inside the band (rare)
                    if (__any_sync(full, band) && band) {
                        double d64[3];
                        in = sep64<2>(G, xpos, n, s, j, d64) < rc2;
                    }
                    const unsigned bal = __ballot_sync(full, in);
                    if (bal) {
                        const int base = __shfl_sync(full, cnt, h);
                        if (in) {
                            const int pos = base + __popc(bal & lt);
                            if (pos < K) lists[(size_t)s * Ks + pos] = ej;
                        }
                        if (lane == h) cnt += __popc(bal);
                    }
                }
            }
            __syncwarp();
        }
        if (lane < nh) {
            const int s = h0 + lane;
            if (cnt > K) {
                atomicOr(B.err, kErrCapacity);
                cnt = K;
            }
            // the row up to a multiple of four (Ks is one): the particle itself
            for (int k = cnt; k & 3; ++k) lists[(size_t)s * Ks + k] = list_entry((uint32_t)s, 13, false);
            B.pcount[s] = cnt;
        }
        __syncwarp();
    }
}

// 2D problems with fewer row segments than this take k_nlist_cells2: a warp per
// cell instead of one per three keeps more warps busy (200 x 200, 1,452 segments:
// a step of ten 0.311 ms, 0.320 ms with k_nlist_home).
constexpr int kRowsMinSegments = 16384;

// Lists with the home particles in the lanes: one warp per row segment of kSeg2
// cells along x in 2D (a 2D cell holds about 9 particles, so three fill most of the
// lanes), per cell in 3D (about 28 particles). Bound by instruction issue.
//  - Staging. The candidates of the surrounding cells pass in the order rows (dz,
//    dy), column, slot; one farther than the cutoff from the whole segment is
//    dropped; the others are moved into the frame of the segment's first cell
//    and packed into shared memory, coordinates by component, entries apart.
//  - Tests. Each lane tests a chunk of 32 candidates against its particle without
//    a branch: t = |r|^2 - lo, two candidates per packed instruction and four per
//    16-byte broadcast read; the sign bit is shifted into the lane's mask word,
//    and the smallest t >= 0 kept as an integer (below the band's width: a
//    candidate inside the band around the cutoff; then the chunk's band
//    candidates take the FP64 test).
//  - Emission. The roles turn round: a lane per candidate, one home particle
//    after the other. The particle's mask word says which lanes write, the bits
//    before a lane's own where, so every hit costs the warp nothing beyond its
//    particle's word and the hits of a chunk leave as one contiguous run. (Each
//    lane walking the bits of its own words: 1.4 times as long at 128^3, the
//    lanes out of step.)
// For every particle the candidates of its own 3^D cells come in the order of
// k_nlist_cells2; the FP32 separation o_i - (o_j + shift s) decides outside the
// band as the canonical form does, so sets and order are the same on every path.
// The FP64 path takes the same pre-test (its offsets are kept for it): FP64 tests
// of every candidate run at 1/64 of the rate (45^3: 3.7 ms a build, now 0.1 ms).
// Against the builders with a per-hit append by the home particle's lane: 128^3
// 2.04 ms a build, now 0.85 ms; the 64-vortex batch 0.37 ms, now 0.24 ms. 61^3: 0.14 ms,
// 96 M warp instructions, 69% of the issue slots.
constexpr int kListWarps = 4;                 // warps per block
constexpr int kStage = 256;                   // staged candidates per warp

// |o_i - c|^2 - lo of a home particle and a staged candidate in the same frame.
template <int D>
__device__ __forceinline__ float near_test(float4 oi, float x, float y, float z, float neg_lo)
{
    const float d0 = __fsub_rn(x, oi.x), d1 = __fsub_rn(y, oi.y);
    float t = __fmaf_rn(d1, d1, __fmaf_rn(d0, d0, neg_lo));
    if (D == 3) {
        const float d2 = __fsub_rn(z, oi.z);
        t = __fmaf_rn(d2, d2, t);
    }
    return t;
}

// near_test of two candidates.
template <int D>
__device__ __forceinline__ void near_test2(const F2 *oi, F2 x, F2 y, F2 z, F2 neg_lo, uint32_t &a, uint32_t &b)
{
    const F2 d0 = sub2(x, oi[0]), d1 = sub2(y, oi[1]);
    F2 t = fma2(d1, d1, fma2(d0, d0, neg_lo));
    if (D == 3) {
        const F2 d2 = sub2(z, oi[2]);
        t = fma2(d2, d2, t);
    }
    float ta, tb;
    unpack2(t, ta, tb);
    a = __float_as_uint(ta);
    b = __float_as_uint(tb);
}

template <int D>
__global__ void __launch_bounds__(kListWarps * kWarp) k_nlist_home(Buffers B, const double *xpos,
                                                                   uint32_t *__restrict__ lists, int Ks)
{
    grid_start<false>();
    if (skip_relist(B)) return;   // (the step graph: relisting or not)
    constexpr int SEG = D == 2 ? kSeg2 : 1;
    constexpr int NCOL = SEG + 2;                       // candidate columns
    constexpr int NT = (D == 3 ? 9 : 3) * NCOL;         // candidate cells
    constexpr int kHomeRow = D == 3 ? 4 : 1;            // the row dy = dz = 0
    __shared__ __align__(16) float cx[kListWarps][D][kStage];
    __shared__ uint32_t ent[kListWarps][kStage];
    // per home particle of the round: its mask word of the chunk, and where its
    // next entry goes from the round's first row (2D: and its cell, bits 30-31)
    __shared__ __align__(16) uint2 word[kListWarps][kWarp];
    __shared__ int own[kListWarps][kWarp];              // staged place of each home particle, -1
    __shared__ int tpre[kListWarps][NT + 1];            // candidates before cell t
    __shared__ int tbeg[kListWarps][NT];                // first slot of cell t
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & (kWarp - 1), w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int g = blockIdx.x * kListWarps + w;          // global segment (2D), cell (3D) of this warp
    if (g >= (D == 2 ? B.nseg2 : B.ncell)) return;      // whole warp
    const int inst = D == 2 ? segment_instance(B, g) : cell_instance(B, g);
    const Geom &G = B.geo[inst];
    const int nx = G.nc[0], ny = G.nc[1], nz = G.nc[2];
    int cx0, cy0, cz0, lc, ns = 1;                      // first cell of the segment, its cells
    if (D == 2) {
        const int nsx = (nx + SEG - 1) / SEG;
        const int ls = g - B.inst[inst].seg_off;
        cx0 = (ls % nsx) * SEG;
        cy0 = ls / nsx;
        cz0 = 0;
        lc = cy0 * nx + cx0;
        ns = min(SEG, nx - cx0);
    } else {
        lc = g - B.inst[inst].cell_off;
        if (lc >= nx * ny * nz) return;                 // the instance's empty sentinel cell
        cx0 = lc % nx;
        cy0 = (lc / nx) % ny;
        cz0 = lc / (nx * ny);
    }
    const int *start = B.cell_start + B.inst[inst].cell_off;
    const int hb = start[lc], he = start[lc + ns];
    if (hb == he) return;
    // first slots of a 2D segment's second and third cells
    const int b1 = D == 2 && ns > 1 ? start[lc + 1] : he, b2 = D == 2 && ns > 2 ? start[lc + 2] : he;
    const float sx = G.s_f[0], sy = G.s_f[1], sz = G.s_f[2];
    const float neg_lo = -G.rc2_lo, box_cut2 = G.rc2_hi * 1.001f, seg_w = (float)ns * sx;
    const uint32_t band = __float_as_uint(G.rc2_hi - G.rc2_lo);
    const int K = B.K, n = B.n;
    // the candidate cells side by side: lane t takes row t / NCOL = (dy + 1) +
    // 3 (dz + 1) and column t % NCOL (x = cx0 - 1 + column); empty when off a closed
    // edge or past the segment's last column
    int m = 0, beg = 0;
    if (lane < NT) {
        const int k = lane % NCOL, r = lane / NCOL;
        int x = cx0 - 1 + k, y = cy0 + r % 3 - 1, z = D == 3 ? cz0 + r / 3 - 1 : 0;
        bool ok = k < ns + 2;
        if (ok && (x < 0 || x >= nx)) { if (G.periodic[0]) x = x < 0 ? x + nx : x - nx; else ok = false; }
        if (ok && (y < 0 || y >= ny)) { if (G.periodic[1]) y = y < 0 ? y + ny : y - ny; else ok = false; }
        if (D == 3 && ok && (z < 0 || z >= nz)) { if (G.periodic[2]) z = z < 0 ? z + nz : z - nz; else ok = false; }
        if (ok) {
            const int nc = (z * ny + y) * nx + x;
            beg = start[nc];
            m = start[nc + 1] - beg;
        }
        tbeg[w][lane] = beg;
    }
    int incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane < NT) tpre[w][lane] = incl - m;
    const int total = __shfl_sync(full, incl, NT - 1);
    if (lane == 0) tpre[w][NT] = total;
    const uint32_t bit = 0x80000000u >> lane, before = ~(0xffffffffu >> lane);
    for (int h0 = hb; h0 < he; h0 += kWarp) {
        const int s = h0 + lane;
        const bool act = s < he;
        const int nh = min(kWarp, he - h0);
        const int kh = D == 2 ? (s >= b1) + (s >= b2) : 0;      // the lane's cell in the segment
        // NaN fails every test whatever the scale of the coordinates (its bits are those
        // of a large positive number: arithmetic gives 0x7fffffff): an idle lane's place,
        // and below the fill of the last chunk
        const float nan = __int_as_float(0x7fffffff);
        float4 oi = make_float4(nan, nan, nan, 0.f);
        if (act) {
            oi = B.off[s];
            if (D == 2) oi.x = __fadd_rn(oi.x, (float)kh * sx);
        }
        const F2 oi2[3] = {both(oi.x), both(oi.y), both(oi.z)};
        const F2 neg_lo2 = both(neg_lo);
        uint32_t *out0 = lists + (size_t)h0 * Ks;       // the round's first row
        int cnt = 0;                                    // list length so far
        int t = 0;                                      // candidate cell of the next position
        int p0 = 0;                                     // candidates looked at
        int take = 0;                                   // staged, not yet tested
        own[w][lane] = -1;
        __syncwarp();
        do {
            // stage: 32 candidates at a time while they fit
            while (p0 < total && take <= kStage - kWarp) {
                const int p = p0 + lane;
                bool keep = false;
                float ex = 0.f, ey = 0.f, ez = 0.f;
                uint32_t e = 0u;
                int h = -1;                             // a home particle's own place: which
                if (p < total) {
                    while (tpre[w][t + 1] <= p) ++t;
                    const int j = tbeg[w][t] + (p - tpre[w][t]);
                    const float4 oj = B.off[j];
                    const int r = t / NCOL, k = t % NCOL;
                    ex = __fadd_rn(oj.x, (float)(k - 1) * sx);
                    ey = __fadd_rn(oj.y, (float)(r % 3 - 1) * sy);
                    const float bx = fmaxf(fmaxf(-ex, ex - seg_w), 0.f);
                    const float by = fmaxf(fmaxf(-ey, ey - sy), 0.f);
                    float b = bx * bx + by * by;
                    if (D == 3) {
                        ez = __fadd_rn(oj.z, (float)(r / 3 - 1) * sz);
                        const float bz = fmaxf(fmaxf(-ez, ez - sz), 0.f);
                        b += bz * bz;
                    }
                    keep = b < box_cut2;
                    // the shift code (dx + 1) + 3 (dy + 1) + 9 (dz + 1) with the column in
                    // the place of dx + 1: emission takes the home cell's column off it
                    e = list_entry((uint32_t)j, k + 3 * r + (D == 2 ? 9 : 0), oj.w != 0.f);
                    if (r == kHomeRow && k >= 1 && k <= ns && j >= h0 && j < h0 + kWarp) h = j - h0;
                }
                const unsigned bal = __ballot_sync(full, keep);
                if (keep) {
                    const int at = take + __popc(bal & lt);
                    cx[w][0][at] = ex;
                    cx[w][1][at] = ey;
                    if constexpr (D == 3) cx[w][2][at] = ez;
                    ent[w][at] = e;
                    if (h >= 0) own[w][h] = at;
                }
                take += __popc(bal);
                p0 += kWarp;
            }
            const bool end = p0 >= total;
            if (end && (take & (kWarp - 1))) {
                // the last chunk is filled up with candidates that fail every test
                const int at = take + lane;
                take = (take + kWarp - 1) / kWarp * kWarp;
                if (at < take) {
                    cx[w][0][at] = nan;
                    cx[w][1][at] = nan;
                    if constexpr (D == 3) cx[w][2][at] = nan;
                    ent[w][at] = 0u;
                }
            }
            __syncwarp();
            const int mine = own[w][lane];
            const int nfull = take / kWarp;
            for (int c = 0; c < nfull; ++c) {
                uint32_t hits = 0u, near = 0xffffffffu;
                const ulonglong2 *x4 = reinterpret_cast<const ulonglong2 *>(&cx[w][0][c * kWarp]);
                const ulonglong2 *y4 = reinterpret_cast<const ulonglong2 *>(&cx[w][1][c * kWarp]);
                const ulonglong2 *z4 = reinterpret_cast<const ulonglong2 *>(&cx[w][D - 1][c * kWarp]);
#pragma unroll
                for (int q = 0; q < kWarp / 4; ++q) {
                    const ulonglong2 X = x4[q], Y = y4[q], Z = z4[q];
                    uint32_t b[4];                       // candidate i of the chunk: bit 31 - i
                    near_test2<D>(oi2, F2{X.x}, F2{Y.x}, F2{Z.x}, neg_lo2, b[0], b[1]);
                    near_test2<D>(oi2, F2{X.y}, F2{Y.y}, F2{Z.y}, neg_lo2, b[2], b[3]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        hits = __funnelshift_l(b[u], hits, 1);
                        near = min(near, b[u]);
                    }
                }
                // the FP64 decision inside the band (rare)
                if (__any_sync(full, near < band) && near < band) {
                    for (int q = 0; q < kWarp; ++q) {
                        const int at = c * kWarp + q;
                        const float d2 = near_test<D>(oi, cx[w][0][at], cx[w][1][at], cx[w][D - 1][at], neg_lo);
                        if (__float_as_uint(d2) >= band) continue;
                        double d64[3];
                        if (sep64<D>(G, xpos, n, s, entry_slot(ent[w][at]), d64) < G.rc2) hits |= 0x80000000u >> q;
                    }
                }
                if (mine >> 5 == c) hits &= ~(0x80000000u >> (mine & 31));    // not itself
                const int nhit = __popc(hits);
                // (a list longer than its row is cut there and raises the error below)
                word[w][lane] = make_uint2(cnt + nhit <= Ks ? hits : 0u, (uint32_t)(lane * Ks + cnt) | (uint32_t)kh << 30);
                cnt += nhit;
                __syncwarp();
                const uint32_t e = ent[w][c * kWarp + lane];
                const ulonglong2 *wd = reinterpret_cast<const ulonglong2 *>(&word[w][0]);
                auto put = [&](unsigned long long v) {
                    const uint32_t hm = (uint32_t)v, at = (uint32_t)(v >> 32);
                    if (hm & bit) {
                        const uint32_t o = D == 2 ? at & 0x3fffffffu : at;
                        out0[o + __popc(hm & before)] = D == 2 ? e - ((at >> 30) << kCodeShift) : e;
                    }
                };
#pragma unroll 4
                for (int h = 0; h < nh; h += 2) {        // (an idle lane's word is empty)
                    const ulonglong2 v = wd[h >> 1];
                    put(v.x);
                    put(v.y);
                }
                __syncwarp();
            }
            // the candidates of an unfinished chunk move to the front
            const int left = take - nfull * kWarp;
            float fx = 0.f, fy = 0.f, fz = 0.f;
            uint32_t fe = 0u;
            if (lane < left) {
                const int at = nfull * kWarp + lane;
                fx = cx[w][0][at];
                fy = cx[w][1][at];
                fz = cx[w][D - 1][at];
                fe = ent[w][at];
            }
            __syncwarp();
            if (lane < left) {
                cx[w][0][lane] = fx;
                cx[w][1][lane] = fy;
                if constexpr (D == 3) cx[w][2][lane] = fz;
                ent[w][lane] = fe;
            }
            own[w][lane] = mine - nfull * kWarp;        // (tested: negative)
            __syncwarp();
            take = left;
        } while (p0 < total || take > 0);
        if (act) {
            // the row up to a multiple of four (Ks is one): the particle itself
            for (int k = cnt; (k & 3) && k < Ks; ++k) out0[lane * Ks + k] = list_entry((uint32_t)s, 13, false);
            if (cnt > K) {
                atomicOr(B.err, kErrCapacity);
                for (int k = 0; k < Ks; ++k) out0[lane * Ks + k] = list_entry((uint32_t)s, 13, false);
                cnt = K;
            }
            B.pcount[s] = cnt;
        }
        __syncwarp();
    }
}

}  // namespace

static_assert(list_stride(1) % 4 == 0, "a list row holds whole 16-byte stores");

bool nlist_few_cells(const Buffers &B) { return B.dim == 2 && B.nseg2 < kRowsMinSegments; }

// The lists of every slot at xpos (order of the latest binning); one launch.
void launch_nlist(const Buffers &B, const double *xpos, cudaStream_t st)
{
    const int Ks = list_stride(B.K);
    if (nlist_few_cells(B)) {
        const int nb = (B.ncell + kWarpsPerBlock - 1) / kWarpsPerBlock;
        launch_next(B, st, nb, kBlock, k_nlist_cells2, B, xpos, B.pjt, Ks);
    } else if (B.dim == 2) {
        const int nb = (B.nseg2 + kListWarps - 1) / kListWarps;
        launch_next(B, st, nb, kListWarps * kWarp, k_nlist_home<2>, B, xpos, B.pjt, Ks);
    } else {
        const int nb = (B.ncell + kListWarps - 1) / kListWarps;
        launch_next(B, st, nb, kListWarps * kWarp, k_nlist_home<3>, B, xpos, B.pjt, Ks);
    }
}

}  // namespace dtsph
