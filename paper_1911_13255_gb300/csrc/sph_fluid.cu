// Fluid pair loops at h_F (Section 3.1), part 1: momentum (Eq.
// fluid-model-mr-mom) with the low-dissipation Riemann pressure and the
// viscous term, the fluid-solid ghost forces (Eqs. fs-force-mr-sp,
// fs-force-mr-sv with the time-averaged solid state of Eq. fs-coupling-mr),
// their solid-side counterparts (Eqs. F:p, F:v), and the FP64 neighbour-set
// debug kernel.  Shared loop machinery: sph_pairs.cuh.
#include <type_traits>

#include "sph_common.cuh"
#include "sph_pairs.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// a4: equation of state + momentum + kick
// ---------------------------------------------------------------------------
// Also leaves the boundary part of target i's continuity equation at v^{n+1}
// (fs_pair_force) in bnd.
// SETS: what the loop visits; kFluidOnly skips the listed targets (row form).
template <int D, int L, bool CP, int FORM, int SETS>
__device__ __forceinline__ void momentum_one(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int i,
                                                 bool act_, int lane, uint32_t *list, int stride, const TileSrc *ts)
{
    const bool act = act_ && (SETS != kFluidOnly || !(f.nbc[i] & (kListSolid | kListWalls | kListOver))) &&
                     (f.only < 0 || takes(f, f.inst[i]));
    const int b = act ? f.inst[i] : 0;
    const Inst &In = bt.I[b];
    const Grid &g = In.g;
    const Phys &P = In.P;
    unsigned nff = 0, nfw = 0, nfs = 0;
    float acc[3] = {0.f, 0.f, 0.f}, afs[3] = {0.f, 0.f, 0.f}, bnd[4] = {0.f, 0.f, 0.f, 0.f};
    float4 Pi = make_float4(0.f, 0.f, 0.f, 0.f), Vi = Pi;
    if (act) {
        Pi = f.P4[i];
        Vi = f.V4[i];
        const float vi[3] = {Vi.x, Vi.y, Vi.z};
        const float rhoi = P.rho0 + Vi.w, pi = Pi.w;
        int cx, cy, cz;
        cell_xyz<D>(f.cell_of[i], In, cx, cy, cz);
        const float c0 = P.c0, eta2 = 2.0f * P.eta;
        // dW / r = dWcF / h (1 - r / 2h)^3
        const float half_inv_h = 0.5f * P.inv_hF, mdW = P.mF * (P.dWcF * P.inv_hF);
        // walls (v~ = a~ = 0) and solid particles at their start-of-step
        // positions with v~, a~
        auto wall_pair = [&](int a, float ox, float oy, float oz) {
            float d[3];
            float r2 = rel_d<D>(Pi, w.A4[a], ox, oy, oz, d);
            if (r2 >= P.rc2F) return;
            nfw++;
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            float o[3];
            fs_pair_force<D>(d, r2, vi, rhoi, pi, z4, z4, w.N4[a], P.VW, P, o, bnd);
            acc[0] += o[0];
            acc[1] += o[1];
            acc[2] += o[2];
        };
        auto solid_pair = [&](int b, float ox, float oy, float oz) {
            float d[3];
            float r2 = rel_d<D>(Pi, s.A4[b], ox, oy, oz, d);
            if (r2 >= P.rc2F) return;
            nfs++;
            float o[3];
            fs_pair_force<D>(d, r2, vi, rhoi, pi, s.VB4[b], s.AB4[b], s.N4[b], P.VS, P, o, bnd);
            afs[0] += o[0];
            afs[1] += o[1];
            afs[2] += o[2];
        };
        // fluid neighbours: Riemann pressure + viscous (Eq. fluid-model-mr-mom, reading R4)
        nff = fluid_pairs<D, L, CP, FORM, SETS, SETS == kAllSets>(f, w, s, g, In.c0, cx, cy, cz, i, lane, Pi, P.rc2F, list, stride, ts,
                                      [&](int j) { return f.V4[j]; },
                                      [&](int, const float4 &Pj, const float4 &Vj, const float *d, float r2, float,
                                          float, float) {
                // two particles at one FP32 position (a clumped pair): the
                // direction is undefined and the pair's terms vanish with r (a NaN
                // goes through, into the sums)
                if (r2 < kMinNormal) return;
                const float rhoj = P.rho0 + Vj.w;
                const float invr = rsqrt_normal(r2);
                const float a = 1.0f - half_inv_h * (r2 * invr);
                // U_L - U_R = -(v_i - v_j).d / r (e = -d / r points from i to j)
                const float dv[3] = {vi[0] - Vj.x, vi[1] - Vj.y, D == 3 ? vi[2] - Vj.z : 0.0f};
                const float du = -(dv[0] * d[0] + dv[1] * d[1] + (D == 3 ? dv[2] * d[2] : 0.0f)) * invr;
                const float beta = fminf(3.0f * fmaxf(du, 0.0f), c0);
                // 2 P* = p_i + p_j + (rho_i + rho_j) / 2 beta (U_L - U_R)
                const float P2 = (pi + Pj.w) + (0.5f * (rhoi + rhoj)) * (beta * du);
                const float sc = __fdividef(a * a * a * mdW, rhoj);   // V_j dW / r
                acc[0] += sc * (eta2 * dv[0] - P2 * d[0]);
                acc[1] += sc * (eta2 * dv[1] - P2 * d[1]);
                if (D == 3) acc[2] += sc * (eta2 * dv[2] - P2 * d[2]);
            }, wall_pair, solid_pair);
    }
    for (int k = 0; k < D; k++) {
        acc[k] = group_sum<L>(acc[k]);
        if (SETS == kAllSets) afs[k] = group_sum<L>(afs[k]);
        if (SETS != kFluidOnly) bnd[k] = group_sum<L>(bnd[k]);
    }
    if (SETS != kFluidOnly) bnd[3] = group_sum<L>(bnd[3]);
    Counts cnt = {nff, nfw, nfs, 0u, 0.0f, {0.0, 0.0, 0.0}};
    if (act && lane == 0) {
        const float rhoi = P.rho0 + Vi.w;
        const float vi[3] = {Vi.x, Vi.y, Vi.z};
        float inv_rho = 1.0f / rhoi;
        float a[3], vn[3] = {0.f, 0.f, 0.f};
        double dt = bt.ctl[b].dt;
        for (int k = 0; k < D; k++) {
            a[k] = (acc[k] + afs[k]) * inv_rho + P.g[k];
            vn[k] = vi[k] + (float)dt * a[k];
            f.dvdt[(size_t)i * D + k] = a[k];
        }
        f.W4[i] = make_float4(vn[0], vn[1], vn[2], Vi.w);
        if (SETS != kFluidOnly) {
            float r = bnd[3];
            for (int k = 0; k < D; k++) r += bnd[k] * (vn[k] - vi[k]);
            f.bnd[i] = r;
        }
        cnt.vmax = sqrtf(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
        // a position that is no number is in nobody's support where rows or
        // compacted lists are tested with "<": the finish kernel hears of it here
        if (Pi.x != Pi.x || Pi.y != Pi.y || (D == 3 && Pi.z != Pi.z)) cnt.vmax = __int_as_float(0x7fffffff);
        if (SETS == kAllSets) {
            float Vi_ = P.mF / rhoi;   // force = V_i * afs (same V_i as the solid side)
            for (int k = 0; k < D; k++) cnt.mom[k] = (double)(Vi_ * afs[k]);
        }
    }
    flush_counts<D>(bt, b, act, cnt, true);
}

// Row form: three kinds of target in one launch (part_blocks).
// Near (a warp per target): a solid of a quarter of the fluid's spacing puts
// hundreds of particles into a cell; with the 4 lanes of the others such a
// target walks about a thousand candidates per lane, and these few thousand
// targets were the tail of the whole launch.
// Walls (kWallLanes lanes): kept apart so that the loop over the rest, 80 to
// 90 % of the targets, holds no boundary code.
// Registers are capped at 64 (80 in the row-of-cells form): more of them cost
// resident warps, which these latency-bound loops need (2-D valve step 69.8 us
// capped, 73.7 us at 92 registers).
// Measured (3-D duct with a plate of a quarter of the fluid's spacing, stage
// events, all targets alike -> in three kinds): 375k particles 637 -> 384 us,
// 3.0M particles 2.49 -> 1.97 ms; reinitialisation 179 -> 107 us and 847 -> 712 us
// per step.  With four entries per load and the pairs of the reinitialisation in
// FP32 these are now 248 us, 1.76 ms, 81 us and 495 us.
template <int D, int L, bool CP, bool TILE, int FORM>
__global__ void __launch_bounds__(kMaxBlock, FORM == 1 ? 3 : 4) k_momentum(Batch bt, Fluid f, Walls w, Solid s)
{
    pdl_enter();
    if (step_failed(bt)) return;   // the step's cell starts are not valid
    extern __shared__ __align__(16) uint8_t s_dyn[];
    uint32_t *const list = (uint32_t *)s_dyn + threadIdx.x;
    const int stride = blockDim.x;
    if constexpr (FORM == 3) {
        const int nn = part_blocks(f.n, kPartNear, blockDim.x), nw = part_blocks(f.n, kPartWall, blockDim.x);
        const int k = blockIdx.x;
        if (k < nn) {
            part_loop<32>(f, kPartNear, k, nn, [&](int i, bool act, int lane) {
                momentum_one<D, 32, CP, FORM, kAllSets>(bt, f, w, s, i, act, lane, nullptr, 0, nullptr);
            });
        } else if (k < nn + nw) {
            part_loop<kWallLanes>(f, kPartWall, k - nn, nw, [&](int i, bool act, int lane) {
                momentum_one<D, kWallLanes, CP, FORM, kFluidWall>(bt, f, w, s, i, act, lane, nullptr, 0, nullptr);
            });
        } else {
            const int t = (k - nn - nw) * blockDim.x + threadIdx.x;
            momentum_one<D, L, CP, FORM, kFluidOnly>(bt, f, w, s, t / L, t / L < f.n, t % L, nullptr, 0, nullptr);
        }
    } else if constexpr (!TILE) {
        const int t = blockIdx.x * blockDim.x + threadIdx.x;
        momentum_one<D, L, CP, FORM, kAllSets>(bt, f, w, s, t / L, t / L < f.n, t % L, list, stride, nullptr);
    } else {
        tile_loop<D, L>(bt, f, f.V4, s_dyn + (CP ? (size_t)kListBytes * blockDim.x : 0),
                        [&](int i, bool act, const TileSrc *ts) {
                            momentum_one<D, L, CP, FORM, kAllSets>(bt, f, w, s, i, act, (int)threadIdx.x % L, list,
                                                                   stride, ts);
                        });
    }
}

int launch_momentum(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int dim, cudaStream_t st)
{
    if (f.n == 0) return 0;
    if (f.n >= kMaxPairTargets) return -7;
    const int parts = f.list ? part_blocks(f.n, kPartNear, f.block) + part_blocks(f.n, kPartWall, f.block) : 0;
    SPH_LAUNCH_PAIRS(k_momentum, f.n, parts, kAllBlocks, bt, f, w, s);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// a2 (neighbour rows): each fluid target's in-support fluid neighbours (from
// the front of its row) and in-support wall neighbours (from the back), in
// the order of the 3^d cells around its cell, with the pair loops' own FP32
// test on the records, and whether a neighbour cell holds solid particles.
// Entries that do not fit are dropped and the row is marked overflowed (its
// target then takes the cell form; every write stays inside the row).  Runs on
// rebuild steps.
// ---------------------------------------------------------------------------
// Row i's word (row_word); a row with boundary neighbours, or one that
// overflowed, also enters the list of its kind (row_part), one atomic per warp and kind (the order of a
// list does not matter: every target is summed by its own lanes).
__device__ __forceinline__ void row_part(const Fluid &f, int i, uint32_t word)
{
    const int kind = word & (kListSolid | kListOver) ? kPartNear : (word & kListWalls ? kPartWall : -1);
    const unsigned here = __activemask();
    const int lane = threadIdx.x & 31;
    for (int p = 0; p < 2; p++) {
        const unsigned m = __ballot_sync(here, kind == p);
        if (kind != p) continue;
        const int lead = __ffs(m) - 1;
        int base = 0;
        if (lane == lead) base = atomicAdd(f.part_n + p, __popc(m));
        base = __shfl_sync(m, base, lead);
        f.part[p][base + __popc(m & ((1u << lane) - 1u))] = i;
    }
}
__device__ __forceinline__ void row_word(const Fluid &f, int i, int nF, int nW, bool solid)
{
    const bool over = nF + nW > f.list_cap || nF > (int)kListCountMask || nW > (int)kListCountMask;
    const uint32_t word =
        kListBuilt | (over ? kListOver : ((uint32_t)nF | ((uint32_t)nW << 11) | (solid ? kListSolid : 0u)));
    f.nbc[i] = word;
    row_part(f, i, word);
}

// The lists again from words that came from elsewhere (a restored state).
__global__ void k_row_parts(Fluid f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < f.n) row_part(f, i, f.nbc[i]);
}

int launch_row_parts(const Fluid &f, cudaStream_t st)
{
    if (f.n == 0) return 0;
    if (cudaMemsetAsync(f.part_n, 0, 2 * sizeof(int), st) != cudaSuccess) return -3;
    k_row_parts<<<(f.n + 255) / 256, 256, 0, st>>>(f);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// One warp per cell, in two stages:
//  - the candidates of the 3^d cells around it, 32 at a time, are tested
//    against the bounding box of the cell's particles (a coalesced load and a
//    ballot) and the ones within reach of it, about 60 % of them, are kept in
//    shared memory in candidate order;
//  - up to kCand of them per lane go to registers, and every particle of the cell is
//    tested against 32 of them per step; a ballot gives the in-support ones
//    consecutive places in its row.
// What bounds a row build is instruction issue over the candidate tests (475
// per particle in 3-D, 61 in 2-D).  With one lane per particle of the cell, as
// this build had it before, 20 to 45 % of the lanes idled (cells of 8 to 18
// particles), every candidate was tested, and each append stored 4 bytes to as
// many rows as lanes; with 8 lanes per particle every particle loaded its
// candidates itself.  Here all lanes test, and a row is written in runs.
// Measured (lane per particle, 8 lanes per particle, this): 3-D duct, 3.0M
// particles, 2052, -, 1172 us; 375k 394, 739, 164 us; 3-D tank, 62k 168, 144,
// 47 us; batch of 32 2-D channels, 577k 124, 234, 109 us; 2-D channel, 10k 22,
// 14, 12 us.  3-D: 127M warp instructions on the 375k duct against 227M, issue
// 65 % active; 4 candidates per lane (96 registers) beat 6 (1714 us on 3.0M) and
// a cap of 80 registers (1290 us).
// The in-support test is the pair loops' own (rel_d on the records).
template <int D> constexpr int kCand = D == 3 ? 4 : 2;   // candidates per lane and batch
constexpr int kRowWarps = 4;

template <int D>
struct RowWarp {
    float4 cand[32 * (kCand<D> + 1)];   // position in its own cell, entry bits
    float4 target[32];
};

__device__ __forceinline__ unsigned ordered_bits(float x)
{
    const unsigned u = __float_as_uint(x);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float from_ordered(unsigned u)
{
    return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}

// Tests the nt targets (slots t0 ..) against the m candidates of the buffer, NR
// of them per lane (straight-line code: the NR tests of a target overlap), and
// appends to their rows; lane t holds target t's count.  WALL: rows are filled
// from the back; otherwise the target itself is left out (entry `self` with
// its slot).
template <int D, bool WALL, int NR>
__device__ __forceinline__ void row_tests(const Fluid &f, const Grid &g, float rc2, const RowWarp<D> &sw, int m, int t0,
                                          int nt, int lane, uint32_t self, int &count)
{
    float4 c[NR];
    float o[NR][3];
#pragma unroll
    for (int r = 0; r < NR; r++) {
        const int k = 32 * r + lane;
        // no candidate: too far for every target
        c[r] = k < m ? sw.cand[k] : make_float4(1e30f, 1e30f, 1e30f, __uint_as_float(0u));
        row_offset(__float_as_uint(c[r].w), g, o[r][0], o[r][1], o[r][2]);
    }
    const unsigned below = (1u << lane) - 1u;
    const int cap = f.list_cap;
    uint32_t *row = f.nbl + (size_t)t0 * cap + (WALL ? cap - 1 : 0);
    uint32_t me = ((uint32_t)t0 << kCodeBits) | self;
#pragma unroll 1
    for (int t = 0; t < nt; t++, row += cap, me += 1u << kCodeBits) {
        const float4 P = sw.target[t];
        int base = __shfl_sync(0xffffffffu, count, t);
        unsigned hit[NR];
#pragma unroll
        for (int r = 0; r < NR; r++) {
            float d[3];
            const bool in = rel_d<D>(P, c[r], o[r][0], o[r][1], o[r][2], d) < rc2 &&
                            (WALL || __float_as_uint(c[r].w) != me);
            hit[r] = __ballot_sync(0xffffffffu, in);
        }
#pragma unroll
        for (int r = 0; r < NR; r++) {
            const int q = base + __popc(hit[r] & below);
            if ((hit[r] >> lane & 1u) && q < cap) row[WALL ? -q : q] = __float_as_uint(c[r].w);
            base += __popc(hit[r]);
        }
        if (lane == t) count = base;
    }
}

template <int D, bool WALL>
__device__ __forceinline__ void row_batch(const Fluid &f, const Grid &g, float rc2, const RowWarp<D> &sw, int m, int t0,
                                          int nt, int lane, uint32_t self, int &count)
{
    const int n = (m + 31) >> 5;
    if constexpr (D == 3) {
        if (n == 4) row_tests<D, WALL, 4>(f, g, rc2, sw, m, t0, nt, lane, self, count);
        else if (n == 3) row_tests<D, WALL, 3>(f, g, rc2, sw, m, t0, nt, lane, self, count);
    }
    if (n == 2) row_tests<D, WALL, 2>(f, g, rc2, sw, m, t0, nt, lane, self, count);
    else if (n == 1) row_tests<D, WALL, 1>(f, g, rc2, sw, m, t0, nt, lane, self, count);
}

template <int D>
__global__ void __launch_bounds__(32 * kRowWarps, D == 3 ? 5 : 8) k_pairlist_cells(Batch bt, Fluid f, Walls w, Solid s)
{
    __shared__ RowWarp<D> s_warp[kRowWarps];
    pdl_enter();
    if (step_failed(bt)) return;   // the step's cell starts are not valid
    if (!rebuild_step(bt, f)) return;
    const int cell = blockIdx.x * kRowWarps + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (cell >= bt.ncell) return;
    const int a0 = f.cstart[cell], a1 = f.cstart[cell + 1];
    if (a0 >= a1) return;
    RowWarp<D> &sw = s_warp[threadIdx.x >> 5];
    const Inst &In = bt.I[f.inst[a0]];
    if (!takes(f, f.inst[a0])) {
        if (a0 == In.f0 && lane == 0) f.nbc[a0] = 0u;   // no rows of this configuration
        return;
    }
    const Grid &g = In.g;
    const float rc2 = In.P.rc2F, reach2 = rc2 * 1.0001f;   // the box test's rounding stays within the margin
    constexpr int NR = D == 3 ? 9 : 3;
    constexpr uint32_t self = 1u | 1u << 2 | 1u << 4;   // the code of the target's own cell
    // lane r < NR: row r's three cells in the fluid, wall and solid sets
    Row3 mf{0, 0, 0, 0, 0, 0}, mw = mf;
    bool solid = false;
    {
        int cx, cy, cz;
        cell_xyz<D>(cell, In, cx, cy, cz);
        const int dy = lane % 3 - 1, dz = D == 3 ? lane / 3 - 1 : 0;
        const int y = cy + dy, z = cz + dz;
        if (lane < NR && y >= 0 && y < g.nc[1] && z >= 0 && z < g.nc[2]) {
            const int base = In.c0 + g.nc[0] * (y + g.nc[1] * z);
            int c[3];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                int x = cx + k - 1;
                if (x < 0 || x >= g.nc[0]) x = g.periodic_x ? (x < 0 ? x + g.nc[0] : x - g.nc[0]) : -1;
                c[k] = x < 0 ? -1 : base + x;
            }
            mf = row_of(f.cstart, c);
            mw = row_of(w.cstart, c);
            if (s.n) solid = row_of(s.cstart, c).n > 0;
        }
        solid = __any_sync(0xffffffffu, solid);
    }
    for (int t0 = a0; t0 < a1; t0 += 32) {
        const int nt = min(32, a1 - t0);
        const float4 P = f.P4[t0 + (lane < nt ? lane : 0)];
        __syncwarp();
        sw.target[lane] = P;
        float lo[3], hi[3];
        {
            const float p[3] = {P.x, P.y, P.z};
#pragma unroll
            for (int k = 0; k < D; k++) {
                lo[k] = from_ordered(__reduce_min_sync(0xffffffffu, ordered_bits(p[k])));
                hi[k] = from_ordered(__reduce_max_sync(0xffffffffu, ordered_bits(p[k])));
            }
        }
        int nF = 0, nW = 0;   // of target `lane`
        auto gather = [&](const Row3 &mine, const float4 *__restrict__ rec, auto wall, int &count) {
            constexpr bool WALL = decltype(wall)::value;
            int m = 0;
            for (int r = 0; r < NR; r++) {
                Row3 row;
                row.n = __shfl_sync(0xffffffffu, mine.n, r);
                if (row.n == 0) continue;
                row.a0 = __shfl_sync(0xffffffffu, mine.a0, r);
                row.a1 = __shfl_sync(0xffffffffu, mine.a1, r);
                row.a2 = __shfl_sync(0xffffffffu, mine.a2, r);
                row.n0 = __shfl_sync(0xffffffffu, mine.n0, r);
                row.n01 = __shfl_sync(0xffffffffu, mine.n01, r);
                const float oy = (float)(1 - r % 3) * g.csf[1], oz = D == 3 ? (float)(1 - r / 3) * g.csf[2] : 0.0f;
                const uint32_t code = (uint32_t)(r % 3) << 2 | (D == 3 ? (uint32_t)(r / 3) : 1u) << 4;
                for (int q0 = 0; q0 < row.n; q0 += 32) {
                    const int q = q0 + lane;
                    int k;
                    const int j = row_slot(row, q < row.n ? q : 0, k);
                    const float4 X = rec[j];
                    // distance of the candidate, in the target cell's frame, from the box
                    const float x = X.x - row_ox(k, g), y = X.y - oy;
                    const float ex = fmaxf(fmaxf(lo[0] - x, x - hi[0]), 0.0f);
                    const float ey = fmaxf(fmaxf(lo[1] - y, y - hi[1]), 0.0f);
                    float e2 = ex * ex + ey * ey;
                    if (D == 3) {
                        const float z = X.z - oz;
                        const float ez = fmaxf(fmaxf(lo[2] - z, z - hi[2]), 0.0f);
                        e2 += ez * ez;
                    }
                    const bool keep = q < row.n && e2 < reach2;
                    const unsigned mk = __ballot_sync(0xffffffffu, keep);
                    if (keep)
                        sw.cand[m + __popc(mk & ((1u << lane) - 1u))] =
                            make_float4(X.x, X.y, X.z, __uint_as_float(((uint32_t)j << kCodeBits) | code | (uint32_t)k));
                    m += __popc(mk);
                    if (m >= 32 * kCand<D>) {
                        __syncwarp();
                        row_batch<D, WALL>(f, g, rc2, sw, 32 * kCand<D>, t0, nt, lane, self, count);
                        m -= 32 * kCand<D>;
                        const float4 rest = sw.cand[32 * kCand<D> + lane];
                        __syncwarp();
                        if (lane < m) sw.cand[lane] = rest;
                    }
                }
            }
            __syncwarp();
            row_batch<D, WALL>(f, g, rc2, sw, m, t0, nt, lane, self, count);
            __syncwarp();
        };
        gather(mf, f.P4, std::false_type{}, nF);
        if (__any_sync(0xffffffffu, mw.n > 0)) gather(mw, w.A4, std::true_type{}, nW);
        if (lane < nt) row_word(f, t0 + lane, nF, nW, solid);
    }
}

int launch_pairlist(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int dim, cudaStream_t st)
{
    if (f.n == 0 || !f.list) return 0;
    if (f.n >= kMaxPairTargets || w.n >= kMaxPairTargets) return -7;
    const unsigned grid = (unsigned)((bt.ncell + kRowWarps - 1) / kRowWarps);
    if (dim == 2) launch_k(k_pairlist_cells<2>, grid, 32 * kRowWarps, 0, st, bt, f, w, s);
    else launch_k(k_pairlist_cells<3>, grid, 32 * kRowWarps, 0, st, bt, f, w, s);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// a5: fluid force on each solid particle, f_a^F = -sum_i V_i (pair term),
// the same pair expression and inputs as a4 (fluid at r^{n+1/2}, v^n)
// ---------------------------------------------------------------------------
template <int D, int L>
__global__ void __launch_bounds__(kMaxBlock, 2) k_solid_fluid_force(Batch bt, Fluid f, Solid s)
{
    pdl_enter();
    if (step_failed(bt)) return;   // the step's cell starts are not valid
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = t / L, lane = t % L;
    const bool act = k < s.n;
    unsigned nsf = 0;
    float fa[3] = {0.f, 0.f, 0.f};
    const int a = act ? __float_as_int(s.N4[k].w) : 0;
    const int b = act ? s.inst[a] : 0;
    const Inst &In = bt.I[b];
    const Grid &g = In.g;
    const Phys &P = In.P;
    if (act) {
        const float4 A = s.A4[k], VB = s.VB4[k], AB = s.AB4[k], N = s.N4[k];
        int cx, cy, cz;
        cell_xyz<D>(s.cell_of[k], In, cx, cy, cz);
        auto pair = [&](int j, float ox, float oy, float oz) {
            const float4 Pj = f.P4[j];
            // the fluid side sees this pair with the opposite cell offset
            float d[3] = {(Pj.x - A.x) - ox, (Pj.y - A.y) - oy, D == 3 ? (Pj.z - A.z) - oz : 0.0f};
            const float r2 = square_norm<D>(d);
            if (r2 >= P.rc2F) return;
            nsf++;
            const float4 Vj = f.V4[j];
            const float vj[3] = {Vj.x, Vj.y, Vj.z};
            const float rhoj = P.rho0 + Vj.w;
            float o[3];
            fs_pair_force<D>(d, r2, vj, rhoj, Pj.w, VB, AB, N, P.VS, P, o);
            float Vf = P.mF / rhoj;
            fa[0] -= Vf * o[0];
            fa[1] -= Vf * o[1];
            fa[2] -= Vf * o[2];
        };
        if (f.reach == 1) {
            // a row of neighbour cells at a time (their starts loaded together)
            for_each_row<D>(g, In.c0, cx, cy, cz, [&](const int c[3], float oy, float oz, int) {
                const Row3 r = row_of(f.cstart, c);
                for (int q = lane; q < r.n; q += L) {
                    int k;
                    const int j = row_slot(r, q, k);
                    pair(j, row_ox(k, g), oy, oz);
                }
            });
        } else {
            for_each_cell<D, 2>(g, In.c0, cx, cy, cz, [&](int c, float ox, float oy, float oz, int) {
                const int j1 = f.cstart[c + 1];
                for (int j = f.cstart[c] + lane; j < j1; j += L) pair(j, ox, oy, oz);
            });
        }
    }
    for (int q = 0; q < D; q++) fa[q] = group_sum<L>(fa[q]);
    Counts cnt = {0u, 0u, 0u, nsf, 0.0f, {0.0, 0.0, 0.0}};
    if (act && lane == 0) {
        for (int q = 0; q < 3; q++) s.fF[3 * a + q] = q < D ? fa[q] : 0.0f;
        for (int q = 0; q < D; q++) cnt.mom[q] = (double)fa[q];
    }
    flush_counts<D>(bt, b, act, cnt, false);
}

// lanes per solid particle of this loop, its own choice: 16 for small
// bodies, whose few particles then spread over more SMs (measured: 2-D dam
// break 12.8 -> 11.1 us), 4 for large ones (batches), where 16 doubles the
// loop's time
constexpr int kSfBlock = 128, kSfSmall = 32768;

int launch_solid_fluid_force(const Batch &bt, const Fluid &f, const Solid &s, int dim, cudaStream_t st)
{
    if (s.n == 0 || f.n == 0) {
        if (s.n) cudaMemsetAsync(s.fF, 0, sizeof(float) * 3 * s.n, st);
        return cudaGetLastError() == cudaSuccess ? 0 : -3;
    }
    const bool small = s.n < kSfSmall;
    if (dim == 2) {
        if (small) launch_k(k_solid_fluid_force<2, 16>, grid_blocks(s.n, 16, kSfBlock), kSfBlock, 0, st, bt, f, s);
        else launch_k(k_solid_fluid_force<2, 4>, grid_blocks(s.n, 4, kSfBlock), kSfBlock, 0, st, bt, f, s);
    } else {
        if (small) launch_k(k_solid_fluid_force<3, 16>, grid_blocks(s.n, 16, kSfBlock), kSfBlock, 0, st, bt, f, s);
        else launch_k(k_solid_fluid_force<3, 4>, grid_blocks(s.n, 4, kSfBlock), kSfBlock, 0, st, bt, f, s);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// Neighbour sets with the FP64 in-support test (debug entry point).  Rows are
// fluid particles (which 0..2, cell-ordered mid-step copy s[1]) or solid
// particles (which 3); counts/fill two-phase; ids in original order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double r2_fp64(double dx, double dy, double dz, int D)
{
    double r2 = __dmul_rn(dx, dx);
    r2 = __dadd_rn(r2, __dmul_rn(dy, dy));
    if (D == 3) r2 = __dadd_rn(r2, __dmul_rn(dz, dz));
    return r2;
}

template <int D>
__global__ void k_debug_pairs(Batch bt, Fluid f, Walls w, Solid s, int inst, int which, int *counts,
                              const int *offs, int *out)
{
    const Inst &In = bt.I[inst];
    const Grid &g = In.g;
    const Phys &P = In.P;
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    int nrows = which == 3 ? In.ns : In.nf;
    if (r >= nrows) return;
    double xi, yi, zi;
    int row, key;
    const FluidState M = f.s[1];
    const int k = (which == 3 ? In.s0 : In.f0) + r;   // sorted slot
    if (which == 3) {
        int a = __float_as_int(s.N4[k].w);   // solid particle of sorted slot k
        xi = s.x[a];
        yi = s.y[a];
        zi = D == 3 ? s.z[a] : 0.0;
        row = a - In.s0;
        key = s.cell_of[k];
    } else {
        xi = M.x[k];
        yi = M.y[k];
        zi = D == 3 ? M.z[k] : 0.0;
        row = M.id[k];
        key = f.cell_of[k];
    }
    int cx, cy, cz;
    cell_xyz<D>(key, In, cx, cy, cz);
    int cnt = 0;
    int base = out ? offs[row] : 0;
    auto visit = [&](int c, float, float, float, int) {
        int j0, j1;
        if (which == 0 || which == 3) {
            j0 = f.cstart[c];
            j1 = f.cstart[c + 1];
        } else if (which == 1) {
            j0 = w.cstart[c];
            j1 = w.cstart[c + 1];
        } else {
            j0 = s.cstart[c];
            j1 = s.cstart[c + 1];
        }
        for (int j = j0; j < j1; j++) {
            double xj, yj, zj;
            int col;
            if (which == 0 || which == 3) {
                if (which == 0 && j == k) continue;
                xj = M.x[j];
                yj = M.y[j];
                zj = D == 3 ? M.z[j] : 0.0;
                col = M.id[j];
            } else if (which == 1) {
                int a = w.perm[j];
                xj = w.x[a];
                yj = w.y[a];
                zj = D == 3 ? w.z[a] : 0.0;
                col = a - In.w0;
            } else {
                int a = __float_as_int(s.N4[j].w);
                xj = s.x[a];
                yj = s.y[a];
                zj = D == 3 ? s.z[a] : 0.0;
                col = a - In.s0;
            }
            double dx = xi - xj;
            if (g.periodic_x) {
                if (dx > 0.5 * g.Lx) dx -= g.Lx;
                else if (dx < -0.5 * g.Lx) dx += g.Lx;
            }
            if (r2_fp64(dx, yi - yj, zi - zj, D) < P.rc2F_d) {
                if (out) out[base + cnt] = col;
                cnt++;
            }
        }
    };
    if (f.reach == 2) for_each_cell<D, 2>(g, In.c0, cx, cy, cz, visit);
    else for_each_cell<D, 1>(g, In.c0, cx, cy, cz, visit);
    if (!out) counts[row] = cnt;
}

int launch_debug_pairs(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int dim, int inst,
                       int which, int *counts, int *offs, int *out, cudaStream_t st)
{
    int nrows = which == 3 ? s.n : f.n;   // upper bound of the instance's rows
    if (nrows == 0) return 0;
    int nb = (nrows + kBlock - 1) / kBlock;
    if (dim == 2) k_debug_pairs<2><<<nb, kBlock, 0, st>>>(bt, f, w, s, inst, which, counts, offs, out);
    else k_debug_pairs<3><<<nb, kBlock, 0, st>>>(bt, f, w, s, inst, which, counts, offs, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace sph
