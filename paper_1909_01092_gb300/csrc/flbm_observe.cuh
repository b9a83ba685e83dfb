// Observables of a state (declared in include/flbm.h as flbm_observables):
// masses, momentum and kinetic energy over the fluid nodes, and the sums
// behind the mode, interdiffusion and momentum temperatures over the bulk
// fluid nodes (arXiv:1909.01092, Section 2, fluctuation-dissipation).
//
// One pass reads every population once. A block of 128 threads walks a column
// of nodes over K planes and keeps its sums in registers; a second launch
// adds the blocks' sums. FP64 is scarce on this GPU (a warp's FP64 instruction
// holds an SM's pipe for about 16 clocks, a float one for a quarter), and the
// sums take some 300 FP64 operations a node and as many again in reductions,
// so the pass works on double-floats (flbm_df.h; both components per packed
// operation where they go alike): linear sums of populations are exact there
// as long as the populations of a node span fewer than 2^24, and a square
// keeps 48 bits, with rounding errors of either sign, so that a sum over
// thousands of nodes is as good as the FP64 one. A block that meets a node
// outside the range this holds for (a population that is not finite or above
// 2^14, a component's density below 2^-30 but not zero) marks itself, and
// k_obs_fp64 redoes it in FP64. A call on 128x128x128 takes 0.34 ms, against
// 3.6 ms with every node in FP64 and 40 full reductions per tile (relative
// errors against FP64 sums in another order: up to 5e-16 both).
#pragma once

#include <algorithm>

#include "flbm_df.h"
#include "flbm_kernels.cuh"

namespace flbm {

// Slots of a block's sums, two values each (x, y):
//   k - 4 for k = 4..18: n_Ak^2, n_Bk^2 (bulk)   15: rho_A, rho_B (bulk)
//   16: rho_A, rho_B (fluid)   17, 18, 19: d_a^2 (bulk), j_a^2 (bulk), a = x, y, z
//   20: rho_A rho_B / rho_tot (bulk), j^2 / (2 rho_tot) (fluid)
//   21: j_x, j_y (fluid)   22: j_z (fluid), bulk nodes   23: non-finite populations
constexpr int kObsSlots = 24;
constexpr int kObsValues = 2 * kObsSlots;
constexpr int kObsThreads = 128;
constexpr float kObsScale = 1099511627776.0f;  // 2^40: keeps squares of modes clear of the float range's ends

// Blocks: column (bx, by) of tx x rows nodes, planes c K .. c K + K - 1.
struct ObsGeom {
    int rows, gy, K, nz;
    long long blocks;  // grid: columns (x fastest) by chunks of planes
};

inline ObsGeom obs_geom(const KParams& P)
{
    ObsGeom g;
    g.rows = kObsThreads / P.tx;
    g.gy = (P.ly + g.rows - 1) / g.rows;
    // Two planes where that leaves four blocks for each of the two an SM
    // holds. No more: the lowest bits of a square are 00 or 01, so a sum that
    // grows past them rounds them down (1e-15 of it over 13 planes).
    const long long planes = (long long)P.gx * g.gy * P.lz;
    g.K = planes >= 2LL * 152 * 8 ? 2 : 1;
    g.K = std::max(g.K, (P.lz + 65534) / 65535);
    g.nz = (P.lz + g.K - 1) / g.K;
    g.blocks = (long long)P.gx * g.gy * g.nz;
    return g;
}

// What a call brings back to the host.
struct ObsOut {
    double v[kObsValues];
    DevState s;
};

// Double-float pair: one double-float per component.
struct PairDf {
    Pair hi, lo;
};
__device__ __forceinline__ PairDf pdf(Pair v) { return PairDf{v, splat(0.0f)}; }
// a + b of two floats, exactly (Knuth's two-sum)
__device__ __forceinline__ PairDf psum(Pair a, Pair b)
{
    const Pair s = add(a, b), bb = sub(s, a);
    return PairDf{s, add(sub(a, sub(s, bb)), sub(b, bb))};
}
__device__ __forceinline__ PairDf padd(PairDf a, PairDf b)
{
    const PairDf s = psum(a.hi, b.hi);
    const Pair e = add(s.lo, add(a.lo, b.lo));
    const Pair h = add(s.hi, e);
    return PairDf{h, sub(e, sub(h, s.hi))};
}
__device__ __forceinline__ PairDf pscale(PairDf a, float c) { return PairDf{mul(a.hi, splat(c)), mul(a.lo, splat(c))}; }
__device__ __forceinline__ PairDf pneg(PairDf a) { return pscale(a, -1.0f); }
__device__ __forceinline__ PairDf psub(PairDf a, PairDf b) { return padd(a, pneg(b)); }
__device__ __forceinline__ df part(PairDf a, int l) { return l ? df(a.hi.y, a.lo.y) : df(a.hi.x, a.lo.x); }
__device__ __forceinline__ PairDf both(df a, df b) { return PairDf{Pair{a.hi, b.hi}, Pair{a.lo, b.lo}}; }
// acc + a^2 (not renormalised: the low part only collects). The square of
// the low part, up to 2^-48 of the whole and never negative, is added to the
// rounding error of the cross term before it meets larger terms: alone it
// would round away every time, and the sum come out 6e-16 too small. So is
// the square's own low part (e, c, tiny) before it meets the accumulator's.
__device__ __forceinline__ void add_square(PairDf& acc, PairDf a)
{
    const Pair p = mul(a.hi, a.hi), e = mad(a.hi, a.hi, mul(p, splat(-1.0f)));
    const Pair h2 = add(a.hi, a.hi), c = mul(h2, a.lo);
    const Pair tiny = mad(a.lo, a.lo, mad(h2, a.lo, mul(c, splat(-1.0f))));
    const PairDf s = psum(acc.hi, p);
    acc.hi = s.hi;
    acc.lo = add(add(acc.lo, s.lo), add(e, add(c, tiny)));
}
// a^2 for one double-float, in the same way.
__device__ __forceinline__ df square(df a)
{
    const float p = __fmul_rn(a.hi, a.hi), e = __fmaf_rn(a.hi, a.hi, -p);
    const float h2 = __fadd_rn(a.hi, a.hi), c = __fmul_rn(h2, a.lo);
    const float tiny = __fmaf_rn(a.lo, a.lo, __fmaf_rn(h2, a.lo, -c));
    return fast_two_sum(p, __fadd_rn(e, __fadd_rn(c, tiny)));
}
// 1 / a to the last bit or so of a double-float, errors of either sign: with
// q = fl(1 / a.hi) and r = 1 - a q (kept to 2^-72), 1 / a = q (1 + r + r^2 + ...).
__device__ __forceinline__ df reciprocal(df a)
{
    const float q = recip_newton(a.hi);
    const float p = __fmul_rn(a.hi, q), pe = __fmaf_rn(a.hi, q, -p);
    const float c = __fmul_rn(a.lo, q), ce = __fmaf_rn(a.lo, q, -c);
    const df s = two_sum(__fadd_rn(1.0f, -p), -pe);  // 1 - p is exact
    const df r = two_sum(s.hi, -c);
    const float rl = __fmaf_rn(r.hi, r.hi, __fadd_rn(__fadd_rn(r.lo, s.lo), -ce));
    return fast_two_sum(q, __fmaf_rn(q, r.hi, __fmul_rn(q, rl)));
}
// a b for a double-float b the same for both components
__device__ __forceinline__ PairDf pmul(PairDf a, df b)
{
    const Pair bh = splat(b.hi), bl = splat(b.lo);
    const Pair p = mul(a.hi, bh);
    Pair e = mad(a.hi, bh, mul(p, splat(-1.0f)));
    e = mad(a.hi, bl, e);
    e = mad(a.lo, bh, e);
    return PairDf{p, e};
}

// Adds one fluid node to the sums; bulk: also to those over the bulk nodes.
__device__ __forceinline__ void observe_node(const Pair f[19], bool bulk, PairDf acc[kObsSlots])
{
    PairDf odd[9];  // d1 d2 d3 d7 d9 d11 d13 d15 d17
#pragma unroll
    for (int q = 0; q < 9; ++q) odd[q] = psum(f[2 * q + 1], mul(f[2 * q + 2], splat(-1.0f)));
    PairDf J[3];
    PairDf a79 = padd(odd[3], odd[4]), m79 = psub(odd[3], odd[4]);
    PairDf a11 = padd(odd[5], odd[6]), m11 = psub(odd[5], odd[6]);
    PairDf a15 = padd(odd[7], odd[8]), m15 = psub(odd[7], odd[8]);
    const PairDf ax[3] = {padd(a79, a11), padd(m79, a15), padd(m11, m15)};
#pragma unroll
    for (int a = 0; a < 3; ++a) J[a] = padd(odd[a], ax[a]);
    if (bulk) {
#pragma unroll
        for (int a = 0; a < 3; ++a) add_square(acc[6 + a], pscale(psub(ax[a], pscale(odd[a], 2.0f)), kObsScale));
        add_square(acc[9], pscale(psub(a79, a11), kObsScale));
        add_square(acc[10], pscale(psub(a15, m79), kObsScale));
        add_square(acc[11], pscale(psub(m11, m15), kObsScale));
    }
    PairDf s[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) s[q] = psum(f[2 * q + 1], f[2 * q + 2]);
    const PairDf f0 = pdf(f[0]);
    const PairDf sxy = padd(s[3], s[4]), sxz = padd(s[5], s[6]), syz = padd(s[7], s[8]);
    const PairDf s23 = padd(s[1], s[2]), sax = padd(s[0], s23), sxx = padd(sxy, sxz), sdg = padd(sxx, syz);
    const PairDf t = padd(f0, sdg);
    const PairDf rho = padd(t, sax);
    // momentum and densities of the mixture
    df j[3], u[3];
    const df rt = part(rho, 0) + part(rho, 1);
    const df irt = reciprocal(rt);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        j[a] = part(J[a], 0) + part(J[a], 1);
        u[a] = j[a] * irt;
    }
    const df jj = j[0] * u[0] + j[1] * u[1] + j[2] * u[2];  // j^2 / rho_tot
    acc[16] = padd(acc[16], rho);
    acc[21] = padd(acc[21], both(j[0], j[1]));
    if (!bulk) {
        acc[20] = padd(acc[20], both(df(0.0f), jj * 0.5f));
        acc[22] = padd(acc[22], both(j[2], df(0.0f)));
        return;
    }
    acc[15] = padd(acc[15], rho);
    acc[20] = padd(acc[20], both(part(rho, 0) * part(rho, 1) * irt, jj * 0.5f));
    acc[22] = padd(acc[22], both(j[2], df(1.0f)));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const df d = (part(rho, 1) * part(J[a], 0) - part(rho, 0) * part(J[a], 1)) * irt;
        add_square(acc[17 + a], both(d * kObsScale, j[a] * kObsScale));
    }
    const df uxx = square(u[0]), uyy = square(u[1]), uzz = square(u[2]);
    const df uu = uxx + uyy + uzz;
    auto mode = [&](int q, PairDf m, df eq) { add_square(acc[q], pscale(psub(m, pmul(rho, eq)), kObsScale)); };
    const PairDf sq = psub(sxx, pscale(syz, 2.0f)), sr = psub(pscale(s[0], 2.0f), s23);
    const PairDf d23 = psub(s[1], s[2]), dxx = psub(sxy, sxz);
    mode(0, psub(sdg, f0), uu);
    mode(1, padd(sr, sq), uxx * 3.0f - uu);
    mode(2, padd(d23, dxx), uyy - uzz);
    mode(3, psub(s[3], s[4]), u[0] * u[1]);
    mode(4, psub(s[7], s[8]), u[1] * u[2]);
    mode(5, psub(s[5], s[6]), u[0] * u[2]);
    add_square(acc[12], pscale(psub(t, pscale(sax, 2.0f)), kObsScale));
    add_square(acc[13], pscale(psub(sq, sr), kObsScale));
    add_square(acc[14], pscale(psub(dxx, d23), kObsScale));
}

// Are the populations of a node within the range observe_node is exact in?
__device__ __forceinline__ bool observe_in_range(const Pair f[19])
{
    uint32_t top = 0u;
    float ra = 0.0f, rb = 0.0f, na = 0.0f, nb = 0.0f;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        top = max(top, max(__float_as_uint(f[i].x) & 0x7fffffffu, __float_as_uint(f[i].y) & 0x7fffffffu));
        ra += f[i].x;
        rb += f[i].y;
        na += fabsf(f[i].x);
        nb += fabsf(f[i].y);
    }
    const float least = 9.31322574615478515625e-10f;  // 2^-30
    return top < __float_as_uint(16384.0f) && ra + rb > least && (na == 0.0f || fabsf(ra) > least) &&
           (nb == 0.0f || fabsf(rb) > least);
}

// Node (x, y, z): is it fluid, and bulk (no particle node among its neighbours)?
__device__ __forceinline__ void observe_kind(int x, int y, int z, const DevState* __restrict__ st,
                                             const uint8_t* __restrict__ masks, const KParams& P, bool& fluid,
                                             bool& bulk)
{
    fluid = bulk = true;
    if (!P.has_particle) return;
    const int o[3] = {st->box0[0], st->box0[1], st->box0[2]};
    const int B2 = P.B + 2;
    if (!(ranges_meet(x, 1, o[0] - 1, B2, P.lx, P.wall[0]) && ranges_meet(y, 1, o[1] - 1, B2, P.ly, P.wall[1]) &&
          ranges_meet(z, 1, o[2] - 1, B2, P.lz, P.wall[2])))
        return;  // outside the particle box grown by one node
    const uint8_t* mask = masks + (size_t)st->cur * P.B * P.B * P.B;
    fluid = !is_solid(x, y, z, o, mask, P);
    bulk = fluid && solid_neighbours(x, y, z, o, mask, P) == 0u;
}

// One step of the transposed warp sum: lanes exchange halves of their N slots.
template <int N>
__device__ __forceinline__ void observe_fold(PairDf* v, int off)
{
    const bool up = (threadIdx.x & off) != 0;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const PairDf keep = up ? v[k + N / 2] : v[k], send = up ? v[k] : v[k + N / 2];
        PairDf r;
        r.hi.x = __shfl_xor_sync(0xffffffffu, send.hi.x, off);
        r.hi.y = __shfl_xor_sync(0xffffffffu, send.hi.y, off);
        r.lo.x = __shfl_xor_sync(0xffffffffu, send.lo.x, off);
        r.lo.y = __shfl_xor_sync(0xffffffffu, send.lo.y, off);
        v[k] = padd(keep, r);
    }
}

// Sums of the block's values (double) into parts[value * blocks + block].
__device__ __forceinline__ void observe_store(const double v[2], int slot, bool owner, double* __restrict__ parts,
                                              long long blocks, long long block)
{
    __shared__ double s_v[kObsThreads / 32][kObsValues];
    if (owner) {
        s_v[threadIdx.x >> 5][2 * slot] = v[0];
        s_v[threadIdx.x >> 5][2 * slot + 1] = v[1];
    }
    __syncthreads();
    if (threadIdx.x < kObsValues) {
        double a = 0.0;
        for (int w = 0; w < kObsThreads / 32; ++w) a += s_v[w][threadIdx.x];
        parts[threadIdx.x * blocks + block] = a;
    }
}

static __global__ void __launch_bounds__(kObsThreads, 2)
    k_obs(const float* __restrict__ f, const DevState* __restrict__ st, const uint8_t* __restrict__ masks,
          double* __restrict__ parts, int* __restrict__ marked, KParams P, ObsGeom G)
{
    const long long block = blockIdx.x + (long long)gridDim.x * blockIdx.y;
    const int by = blockIdx.x / P.gx, bx = blockIdx.x - by * P.gx;
    const int tx = threadIdx.x & (P.tx - 1), ty = threadIdx.x >> (__ffs(P.tx) - 1);
    const int x = bx * P.tx + tx, y = by * G.rows + ty;
    const int z0 = blockIdx.y * G.K, z1 = min(z0 + G.K, P.lz);
    PairDf acc[kObsSlots];
#pragma unroll
    for (int k = 0; k < kObsSlots; ++k) acc[k] = pdf(splat(0.0f));
    bool in_range = true;
    if (x < P.lx && y < P.ly) {
        for (int z = z0; z < z1; ++z) {
            bool fluid, bulk;
            observe_kind(x, y, z, st, masks, P, fluid, bulk);
            if (!fluid) continue;
            const uint32_t n = (uint32_t)x + (uint32_t)P.lx * ((uint32_t)y + (uint32_t)P.ly * (uint32_t)z);
            Pair v[19];
#pragma unroll
            for (int i = 0; i < 19; ++i)
                v[i] = Pair{__ldg(at(f + P.dirN[i], 4u * n)), __ldg(at(f + P.dirN[19 + i], 4u * n))};
            in_range = in_range && observe_in_range(v);
            observe_node(v, bulk, acc);
        }
    }
    if (threadIdx.x == 0) marked[block] = 0;
    if (__syncthreads_or(!in_range)) {
        if (threadIdx.x == 0) marked[block] = 1;
        return;
    }
    // 24 slots over 32 lanes: 12, 6, 3 (+1), 2, 1 a lane; bits 4..0 of the
    // lane then name the slot.
    observe_fold<24>(acc, 16);
    observe_fold<12>(acc, 8);
    observe_fold<6>(acc, 4);
    acc[3] = pdf(splat(0.0f));
    observe_fold<4>(acc, 2);
    observe_fold<2>(acc, 1);
    const int lane = threadIdx.x & 31;
    const int low = 2 * (lane >> 1 & 1) + (lane & 1);  // 0..3 of the last four
    const int slot = 12 * (lane >> 4) + 6 * (lane >> 3 & 1) + 3 * (lane >> 2 & 1) + low;
    double v[2] = {(double)acc[0].hi.x + (double)acc[0].lo.x, (double)acc[0].hi.y + (double)acc[0].lo.y};
    if (slot < 15 || (slot >= 17 && slot < 20)) {
        constexpr double unscale = 1.0 / ((double)kObsScale * (double)kObsScale);
        v[0] *= unscale;
        v[1] *= unscale;
    }
    observe_store(v, slot, low < 3, parts, G.blocks, block);
}

// The blocks k_obs marked, in FP64.
static __global__ void __launch_bounds__(kObsThreads)
    k_obs_fp64(const float* __restrict__ f, const DevState* __restrict__ st, const uint8_t* __restrict__ masks,
               double* __restrict__ parts, const int* __restrict__ marked, KParams P, ObsGeom G)
{
    const long long block = blockIdx.x + (long long)gridDim.x * blockIdx.y;
    if (!marked[block]) return;
    const int by = blockIdx.x / P.gx, bx = blockIdx.x - by * P.gx;
    const int tx = threadIdx.x & (P.tx - 1), ty = threadIdx.x >> (__ffs(P.tx) - 1);
    const int x = bx * P.tx + tx, y = by * G.rows + ty;
    const int z0 = blockIdx.y * G.K, z1 = min(z0 + G.K, P.lz);
    double acc[kObsValues];
    for (int k = 0; k < kObsValues; ++k) acc[k] = 0.0;
    if (x < P.lx && y < P.ly) {
        for (int z = z0; z < z1; ++z) {
            bool fluid, bulk;
            observe_kind(x, y, z, st, masks, P, fluid, bulk);
            if (!fluid) continue;
            const long long n = x + (long long)P.lx * (y + (long long)P.ly * z);
            double m[2][19];
            for (int l = 0; l < 2; ++l) {
                double fl[19];
                for (int i = 0; i < 19; ++i) {
                    const float v = f[(long long)(19 * l + i) * P.N + n];
                    if (!isfinite(v)) acc[46] += 1.0;
                    fl[i] = (double)v;
                }
                to_modes_t<double>(fl, m[l]);
                acc[32 + l] += m[l][0];
            }
            const double rt = m[0][0] + m[1][0];
            const double j[3] = {m[0][1] + m[1][1], m[0][2] + m[1][2], m[0][3] + m[1][3]};
            acc[42] += j[0];
            acc[43] += j[1];
            acc[44] += j[2];
            acc[41] += rt > 0.0 ? (j[0] * j[0] + j[1] * j[1] + j[2] * j[2]) / (2.0 * rt) : 0.0;
            if (!bulk) continue;
            const double u[3] = {j[0] / rt, j[1] / rt, j[2] / rt};
            const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
            const double eq[6] = {uu, 3.0 * u[0] * u[0] - uu, u[1] * u[1] - u[2] * u[2],
                                  u[0] * u[1], u[1] * u[2], u[0] * u[2]};
            for (int l = 0; l < 2; ++l) {
                for (int k = 4; k < 19; ++k) {
                    const double nk = k <= 9 ? m[l][k] - m[l][0] * eq[k - 4] : m[l][k];
                    acc[2 * (k - 4) + l] += nk * nk;
                }
                acc[30 + l] += m[l][0];
            }
            for (int a = 0; a < 3; ++a) {
                const double d = (m[1][0] * m[0][1 + a] - m[0][0] * m[1][1 + a]) / rt;
                acc[34 + 2 * a] += d * d;
                acc[35 + 2 * a] += j[a] * j[a];
            }
            acc[40] += m[0][0] * m[1][0] / rt;
            acc[45] += 1.0;
        }
    }
    __shared__ double s_red[(kObsThreads / 32) * 8];
    __shared__ double s_out[8];
    for (int c = 0; c < kObsValues / 8; ++c) {
        block_sum8<kObsThreads>(acc + 8 * c, s_red, s_out);
        if (threadIdx.x < 8) parts[(8 * c + threadIdx.x) * G.blocks + block] = s_out[threadIdx.x];
        __syncthreads();
    }
}

// Value blockIdx.x summed over the blocks (fixed order); block 0 also copies
// the particle record, so that one copy brings everything to the host.
static __global__ void __launch_bounds__(256) k_obs_sum(const double* __restrict__ parts, long long blocks,
                                                        const DevState* __restrict__ st, ObsOut* __restrict__ out)
{
    __shared__ double s_w[8];
    double a = 0.0;
    for (long long b = threadIdx.x; b < blocks; b += 256) a += parts[blockIdx.x * blocks + b];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += s_w[w];
        out->v[blockIdx.x] = t;
    }
    if (blockIdx.x == 0) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(st);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&out->s);
        for (int w = threadIdx.x; w < (int)(sizeof(DevState) / 4); w += 256) dst[w] = src[w];
    }
}

// Launches of one reduction on stream s; the result is in *out (device).
inline cudaError_t launch_observe(const float* f, const DevState* st, const uint8_t* masks, double* parts, int* marked,
                                  ObsOut* out, const KParams& P, cudaStream_t s)
{
    const ObsGeom G = obs_geom(P);
    const dim3 grid(P.gx * G.gy, G.nz);
    k_obs<<<grid, kObsThreads, 0, s>>>(f, st, masks, parts, marked, P, G);
    k_obs_fp64<<<grid, kObsThreads, 0, s>>>(f, st, masks, parts, marked, P, G);
    k_obs_sum<<<kObsValues, 256, 0, s>>>(parts, G.blocks, st, out);
    return cudaGetLastError();
}

}  // namespace flbm
