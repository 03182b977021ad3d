// Fluid pair loops at h_F (Section 3.1), part 2: continuity (Eq.
// fluid-model-mr-con) with the second half drift, and the density
// reinitialisation of Alg. 1.  Shared loop machinery: sph_pairs.cuh.
#include <type_traits>

#include "sph_common.cuh"
#include "sph_pairs.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// a6: continuity at (r^{n+1/2}, rho^{n+1/2}, v^{n+1}) + second half drift;
// writes the end-of-step state to s[0] in cell order
// ---------------------------------------------------------------------------
template <int D, int L, bool CP, int FORM>
__device__ __forceinline__ void density_one(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int i,
                                                 bool act_, int lane, uint32_t *list, int stride, const TileSrc *ts)
{
    const bool act = act_ && (f.only < 0 || takes(f, f.inst[i]));
    const int b = act ? f.inst[i] : 0;
    const Inst &In = bt.I[b];
    const Grid &g = In.g;
    const Phys &P = In.P;
    float rate = 0.0f;
    float4 Pi = make_float4(0.f, 0.f, 0.f, 0.f), Wi = Pi;
    if (act) {
        Pi = f.P4[i];
        Wi = f.W4[i];
        const float vi[3] = {Wi.x, Wi.y, Wi.z};
        const float drhoi = Wi.w, rhoi = P.rho0 + Wi.w;
        int cx, cy, cz;
        cell_xyz<D>(f.cell_of[i], In, cx, cy, cz);
        const float half_inv_h = 0.5f * P.inv_hF, mdW = P.mF * (P.dWcF * P.inv_hF);   // as in momentum_one
        const EosDiff dp(drhoi, P);
        auto none = [](int, float, float, float) {};
        fluid_pairs<D, L, CP, FORM, kFluidOnly, true>(f, w, s, g, In.c0, cx, cy, cz, i, lane, Pi, P.rc2F, list, stride, ts,
                                [&](int j) { return f.W4[j]; },
                                [&](int, const float4 &, const float4 &Wj, const float *d, float r2, float, float,
                                    float) {
                if (r2 < kMinNormal) return;   // a clumped pair: no direction, dW(0) = 0 (a NaN goes through)
                const float rhoj = P.rho0 + Wj.w;
                const float r = r2 * rsqrt_normal(r2), a = 1.0f - half_inv_h * r;
                const float dot = (vi[0] - Wj.x) * d[0] + (vi[1] - Wj.y) * d[1] +
                                  (D == 3 ? (vi[2] - Wj.z) * d[2] : 0.0f);
                // (v_i - v~_ij).grad_i W = dW / r [(v_i - v_j).d / 2 + r (p_i - p_j) / ((rho_i + rho_j) c0)]
                const float diff = 0.5f * dot + r * __fdividef(dp(Wj.w), (rhoi + rhoj) * P.c0);
                rate += __fdividef(a * a * a * mdW, rhoj) * diff;
            }, none, none);
    }
    rate = group_sum<L>(rate);
    if (!act || lane != 0) return;
    // walls and solid: the momentum loop's sums (fs_pair_force)
    if (FORM != 3 || (f.nbc[i] & (kListSolid | kListWalls | kListOver))) rate += f.bnd[i];
    const float vi[3] = {Wi.x, Wi.y, Wi.z};
    const float rhoi = P.rho0 + Wi.w;
    float rhodot = 2.0f * rhoi * rate;
    // second half drift (Eq. verlet-first-final) and the new state
    const FluidState M = f.s[1], S = f.s[0];
    double h = 0.5 * bt.ctl[b].dt;
    double x = M.x[i] + h * (double)vi[0];
    double y = M.y[i] + h * (double)vi[1];
    if (g.periodic_x) {
        if (x >= g.x_lo + g.Lx) x -= g.Lx;
        else if (x < g.x_lo) x += g.Lx;
    }
    S.x[i] = x;
    S.y[i] = y;
    S.vx[i] = vi[0];
    S.vy[i] = vi[1];
    if (D == 3) {
        S.z[i] = M.z[i] + h * (double)vi[2];
        S.vz[i] = vi[2];
    }
    S.drho[i] = M.drho[i] + (float)h * rhodot;
    S.rhodot[i] = rhodot;
    S.id[i] = M.id[i];
}

template <int D, int L, bool CP, bool TILE, int FORM>
__global__ void __launch_bounds__(kMaxBlock) k_density(Batch bt, Fluid f, Walls w, Solid s)
{
    pdl_enter();
    if (step_failed(bt)) return;   // the step's cell starts are not valid
    extern __shared__ __align__(16) uint8_t s_dyn[];
    uint32_t *const list = (uint32_t *)s_dyn + threadIdx.x;
    const int stride = blockDim.x;
    if constexpr (!TILE) {
        const int t = blockIdx.x * blockDim.x + threadIdx.x;
        density_one<D, L, CP, FORM>(bt, f, w, s, t / L, t / L < f.n, t % L, list, stride, nullptr);
    } else {
        tile_loop<D, L>(bt, f, f.W4, s_dyn + (CP ? (size_t)kListBytes * blockDim.x : 0),
                        [&](int i, bool act, const TileSrc *ts) {
                            density_one<D, L, CP, FORM>(bt, f, w, s, i, act, (int)threadIdx.x % L, list, stride, ts);
                        });
    }
}

int launch_density(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int dim, cudaStream_t st)
{
    if (f.n == 0) return 0;
    if (f.n >= kMaxPairTargets) return -7;
    SPH_LAUNCH_PAIRS(k_density, f.n, 0, kAllBlocks, bt, f, w, s);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// Density reinitialisation (Alg. 1, every n_reinit steps): rho = rho0 sigma /
// sigma0 with the number density sigma = sum_j W_ij V_j / V_i, self term
// included (reading R16).  rho - rho0 = rho0 (sigma - sigma0) / sigma0 loses
// three to four digits to cancellation, so each W_ij must be good to far
// better than FP32.  FP64 arithmetic is a small fraction of the FP32 rate on
// this GPU; the pair terms are therefore carried as unevaluated sums hi + lo of
// two FP32 numbers (about 44 significant bits), from cell-relative positions
// given that way.  Per-particle sums are finished in FP64.
//
// What bounds the loop is FP32 issue, so the pairs are kept short:
//  - a position's FP32 number is cut at a fixed quantum, 2^-21 of a power of
//    two above the cell edge, and so is the edge's: the differences of the upper
//    and of the lower parts are then exact, one addition each instead of a TwoSum
//    (Knuth), and so is their sum with its remainder (Dekker), to which the
//    differences of the records' remainders are added;
//  - the shape (1 - s)^4 (1 + 4 s), s = r / 2h, takes r as FP32 root s plus
//    Newton remainder; the remainder rides on the lo parts of 1 - s and 1 + 4 s,
//    whose hi parts are exact or one FMA from it (Dekker), and no product is
//    renormalised.
// Measured (general double-float additions and products -> cut parts with one
// FP32 number for lower part and remainder -> this; per step with a
// reinitialisation every third): 3-D duct, 3.0M particles 714 -> 448 -> 494 us,
// 375k 107 -> 75 -> 81, tank of 62k 33 -> 23 -> 23.
// Error of a shape (between 0 and 1) against 64 bits, restated on the CPU over
// 400 000 3-D pairs: 8e-15 rms, 1.6e-13 at most; general double-float
// arithmetic, every operation renormalised, 2e-15 and 2e-14; with the lower parts
// and the remainders in one FP32 number 2.4e-13 and 3e-12.  The density it ends in
// is stored as an FP32 deviation, 6e-8 of it.
// ---------------------------------------------------------------------------
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// What the pairs of one target share: the rounding constant, the edges and
// 1 / (2h)^2 as hi + lo.
template <int D>
struct WendlandPairs {
    float big;                  // x + big - big rounds x to the quantum
    float edge_hi[3], edge_mid[3], edge_lo[3], inv_edge[3];
    ff scale;                   // 1 / (4 h^2)
    float hi[3], mid[3], lo[3]; // the target: upper and lower part of its FP32 position, remainder

    __device__ __forceinline__ void split(const float4 &X, float h[3], float m[3]) const
    {
        const float x[3] = {X.x, X.y, X.z};
#pragma unroll
        for (int k = 0; k < D; k++) {
            h[k] = __fsub_rn(__fadd_rn(x[k], big), big);
            m[k] = __fsub_rn(x[k], h[k]);
        }
    }
    __device__ __forceinline__ WendlandPairs(const Grid &g, const Phys &P, const float4 &Pi, const float4 &Li)
    {
        float most = g.csf[0];
        for (int k = 1; k < D; k++) most = fmaxf(most, g.csf[k]);
        // six times the power of two above the largest edge
        big = 6.0f * __int_as_float(((__float_as_int(most) >> 23) + 1) << 23);
        for (int k = 0; k < D; k++) {
            edge_hi[k] = __fsub_rn(__fadd_rn(g.csf[k], big), big);
            edge_mid[k] = __fsub_rn(g.csf[k], edge_hi[k]);
            edge_lo[k] = g.cslo[k];
            inv_edge[k] = 1.0f / g.csf[k];
        }
        const float ih = 0.5f * P.ihF_hi, il = 0.5f * P.ihF_lo;
        scale.hi = __fmul_rn(ih, ih);
        scale.lo = __fmaf_rn(2.0f * ih, il, __fmaf_rn(ih, ih, -scale.hi));
        split(Pi, hi, mid);
        lo[0] = Li.x, lo[1] = Li.y, lo[2] = Li.z;
    }
    // adds the shape of the pair with the particle at X (+ remainder R) in the
    // cell of offset o to sum; beyond the support (the screen lets pairs up to
    // 1.0001 (2h)^2 pass) it is below 1e-16
    __device__ __forceinline__ void add(ff &sum, const float4 &X, const float4 &R, float ox, float oy, float oz) const
    {
        const float o[3] = {ox, oy, oz}, l[3] = {R.x, R.y, R.z};
        float h[3], m[3], p[3], e = 0.0f, c = 0.0f;
        split(X, h, m);
#pragma unroll
        for (int k = 0; k < D; k++) {
            // o is a small whole number of edges
            const float n = __fsub_rn(__fmaf_rn(o[k], inv_edge[k], 12582912.0f), 12582912.0f);
            const float u = __fmaf_rn(n, edge_hi[k], __fsub_rn(hi[k], h[k]));    // exact
            const float v = __fmaf_rn(n, edge_mid[k], __fsub_rn(mid[k], m[k]));  // exact
            const float w = __fmaf_rn(n, edge_lo[k], __fsub_rn(lo[k], l[k]));
            const float d = __fadd_rn(u, v);
            const float dl = __fadd_rn(__fsub_rn(v, __fsub_rn(d, u)), w);   // |u| >= |v|, or u = 0
            p[k] = __fmul_rn(d, d);
            e = __fadd_rn(e, __fmaf_rn(d, d, -p[k]));
            c = __fmaf_rn(d, dl, c);
        }
        ff r2 = ff_two_sum(p[0], p[1]);
        r2.lo = __fadd_rn(r2.lo, e);
        if (D == 3) {
            const ff q = ff_two_sum(r2.hi, p[2]);
            r2.hi = q.hi;
            r2.lo = __fadd_rn(r2.lo, q.lo);
        }
        r2.lo = __fmaf_rn(2.0f, c, r2.lo);
        // t = s^2, s its root: FP32 root plus the Newton remainder ds
        const float t = __fmul_rn(r2.hi, scale.hi);
        const float tl = __fadd_rn(__fmaf_rn(r2.hi, scale.hi, -t),
                                   __fmaf_rn(r2.hi, scale.lo, __fmul_rn(r2.lo, scale.hi)));
        const float rs = rsqrt_normal(fmaxf(t, 1e-30f));
        const float s = __fmul_rn(t, rs);
        const float ds = __fmul_rn(__fmul_rn(0.5f, rs), __fadd_rn(__fmaf_rn(-s, s, t), tl));
        const float u = __fsub_rn(1.0f, s), ul = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, u), s), ds);
        const float v = __fmaf_rn(4.0f, s, 1.0f);
        const float vl = __fmaf_rn(4.0f, ds, __fmaf_rn(4.0f, s, __fsub_rn(1.0f, v)));
        const float u2 = __fmul_rn(u, u), u2l = __fmaf_rn(__fmaf_rn(2.0f, u, ul), ul, __fmaf_rn(u, u, -u2));
        const float u4 = __fmul_rn(u2, u2), u4l = __fmaf_rn(__fmaf_rn(2.0f, u2, u2l), u2l, __fmaf_rn(u2, u2, -u4));
        const float w = __fmul_rn(u4, v);
        const float wl = __fmaf_rn(u4l, vl, __fmaf_rn(u4l, v, __fmaf_rn(u4, vl, __fmaf_rn(u4, v, -w))));
        const ff q = ff_two_sum(sum.hi, w);
        sum.hi = q.hi;
        sum.lo = __fadd_rn(sum.lo, __fadd_rn(q.lo, wl));
    }
};

// The shape sums of one target over the fluid, the walls and the solid.
struct ShapeSums {
    ff f, w, s;
};

// (each lane's own sum is such a pair: the few additions here add 2^-48 of the
// sum each, as every pair's did)
template <int L>
__device__ __forceinline__ ff group_sum_ff(ff v)
{
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, v.hi, o), l = __shfl_xor_sync(0xffffffffu, v.lo, o);
        const ff t = ff_two_sum(v.hi, h);
        v.hi = t.hi;
        v.lo = __fadd_rn(__fadd_rn(v.lo, l), t.lo);
    }
    return v;
}

// (over its L lanes, in every lane)
template <int D, int L, bool CP, int FORM, int SETS>
__device__ __forceinline__ ShapeSums reinit_pairs(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s,
                                                  int i, bool act, int lane, uint32_t *list, int stride,
                                                  const TileSrc *ts)
{
    ff sF = {0.0f, 0.0f}, sW = {0.0f, 0.0f}, sS = {0.0f, 0.0f};
    if (act) {
        const Inst &In = bt.I[f.inst[i]];
        const Grid &g = In.g;
        const Phys &P = In.P;
        const float screen = P.rc2F * 1.0001f;
        const float4 Pi = f.P4[i], Li = f.L4[i];
        const WendlandPairs<D> shape(g, P, Pi, Li);
        int cx, cy, cz;
        cell_xyz<D>(f.cell_of[i], In, cx, cy, cz);
        auto wall_pair = [&](int q, float ox, float oy, float oz) {
            float d[3];
            const float4 Aq = w.A4[q];
            if (rel_d<D>(Pi, Aq, ox, oy, oz, d) >= screen) return;
            shape.add(sW, Aq, w.L4[q], ox, oy, oz);
        };
        auto solid_pair = [&](int q, float ox, float oy, float oz) {
            float d[3];
            const float4 Aq = s.A4[q];
            if (rel_d<D>(Pi, Aq, ox, oy, oz, d) >= screen) return;
            shape.add(sS, Aq, s.L4[q], ox, oy, oz);
        };
        fluid_pairs<D, L, CP, FORM, SETS, SETS == kAllSets, false>(
            f, w, s, g, In.c0, cx, cy, cz, i, lane, Pi, screen, list, stride, ts, [&](int j) { return f.L4[j]; },
            [&](int, const float4 &Pj, const float4 &Lj, const float *, float, float ox, float oy, float oz) {
                shape.add(sF, Pj, Lj, ox, oy, oz);
            },
            wall_pair, solid_pair);
    }
    return {group_sum_ff<L>(sF), group_sum_ff<L>(sW), SETS == kAllSets ? group_sum_ff<L>(sS) : sS};
}

__device__ __forceinline__ void reinit_finish(const Batch &bt, const Fluid &f, int i, const ShapeSums &v)
{
    const Phys &P = bt.I[f.inst[i]].P;
    const double dF = (double)v.f.hi + (double)v.f.lo, dW = (double)v.w.hi + (double)v.w.lo,
                 dS = (double)v.s.hi + (double)v.s.lo;
    double sigma = P.alphaF_d * (1.0 + dF + P.VW_VF_d * dW + P.VS_VF_d * dS);
    double dr = P.rho0_d * ((sigma - P.sigma0_d) / P.sigma0_d);
    if (P.free_surface && dr < 0.0) dr = 0.0;
    float drho = (float)dr;
    f.s[1].drho[i] = drho;
    f.P4[i].w = eos_p(drho, P);
    f.V4[i].w = drho;
}

// Row form: the targets near solid particles and those of overflowed rows take
// a warp each, in the first blocks (as in k_momentum; the walls, whose pairs
// cost no more than the fluid's here, stay with the rest).  The FP64 end of a
// target's sums runs in whole warps (FP64 takes as long for 4 active lanes as
// for 32; 32 flow channels 57 -> 41 us of a step).  On most steps no instance is
// due: a grid of some 30 waves strides over the targets, so that such a step
// costs a launch and not one block per 32 targets (3-D duct, 3.0M particles:
// 121 us, now 22).  A grid of 4 waves leaves the last one too empty (459 -> 543
// us per step with a reinitialisation every third).
constexpr int kReinitBlocks = 152 * 128;

template <int D, int L, bool CP, bool TILE, int FORM>
__global__ void __launch_bounds__(kMaxBlock, D == 2 && FORM != 1 ? 5 : (D == 3 && FORM == 1 ? 3 : 4)) k_reinit(Batch bt, Fluid f, Walls w, Solid s)
{
    pdl_enter();
    if (step_failed(bt)) return;   // the step's cell starts are not valid
    if (bt.B == 1 && !bt.ctl[0].reinit) return;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    uint32_t *const list = (uint32_t *)s_dyn + threadIdx.x;
    const int stride = blockDim.x, lane = (int)threadIdx.x % L;
    constexpr int SETS = FORM == 3 ? kFluidWall : kAllSets;
    // is this a reinitialisation step of target i's instance?
    auto due = [&](int i) { return i < f.n && bt.ctl[f.inst[i]].reinit && takes(f, f.inst[i]); };
    if constexpr (!TILE) {
        const int nn = FORM == 3 ? part_blocks(f.n, kPartNear, blockDim.x) : 0;
        if ((int)blockIdx.x < nn) {
            part_loop<32>(f, kPartNear, blockIdx.x, nn, [&](int i, bool act, int l) {
                const bool go = act && due(i);
                const ShapeSums v = reinit_pairs<D, 32, CP, FORM, kAllSets>(bt, f, w, s, i, go, l, nullptr, 0, nullptr);
                if (go && l == 0) reinit_finish(bt, f, i, v);
            });
            return;
        }
        __shared__ ShapeSums s_sums[kMaxBlock / L];
        auto mine = [&](int i) {
            return due(i) && (FORM != 3 || !(f.nbc[i] & (kListSolid | kListOver)));
        };
        const int per = blockDim.x / L, k = (int)threadIdx.x / L, step = ((int)gridDim.x - nn) * per;
        for (int i0 = ((int)blockIdx.x - nn) * per; i0 < f.n; i0 += step) {
            const bool act = mine(i0 + k);
            if (!__syncthreads_or(act)) continue;   // no instance of these targets is due
            const ShapeSums v =
                reinit_pairs<D, L, CP, FORM, SETS>(bt, f, w, s, i0 + k, act, lane, list, stride, nullptr);
            if (lane == 0) s_sums[k] = v;
            __syncthreads();
            if ((int)threadIdx.x < per && mine(i0 + threadIdx.x))
                reinit_finish(bt, f, i0 + threadIdx.x, s_sums[threadIdx.x]);
        }
    } else {
        if (!bt.ctl[f.tiles[blockIdx.x].x].reinit) return;   // not a reinitialisation step of this instance
        tile_loop<D, L>(bt, f, f.L4, s_dyn + (CP ? (size_t)kListBytes * blockDim.x : 0),
                        [&](int i, bool act, const TileSrc *ts) {
                            const bool go = act && due(i);
                            const ShapeSums v =
                                reinit_pairs<D, L, CP, FORM, kAllSets>(bt, f, w, s, i, go, lane, list, stride, ts);
                            if (go && lane == 0) reinit_finish(bt, f, i, v);
                        });
    }
}

int launch_reinit(const Batch &bt, const Fluid &f, const Walls &w, const Solid &s, int dim, cudaStream_t st)
{
    if (f.n == 0) return 0;
    if (f.n >= kMaxPairTargets) return -7;
    SPH_LAUNCH_PAIRS(k_reinit, f.n, f.list ? part_blocks(f.n, kPartNear, f.block) : 0, kReinitBlocks, bt, f, w, s);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace sph
