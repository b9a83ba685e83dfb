// The collide-stream kernels and the particle update of one FLBM step
// (arXiv:1909.01092, Section 2: Eq. (lbe), Eq. (sc-force), particle coupling;
// Section 3: Eq. (fp), channel walls).
//
// Tiles (TX x TY nodes of one z-plane, one CTA each) split into two sets:
//   bulk tiles  : no node of the tile or its one-node halo is a particle node;
//                 k_collide_bulk runs them with no particle code at all.
//   near tiles  : the tile meets the particle box grown by one node;
//                 k_collide_near runs them over a fixed grid of candidates
//                 around the box and reduces force, torque and mass ledger.
// Both kernels apply the same tile_near() test, so every tile runs exactly once.
// The particle update runs in the last block of the near launch (after every
// candidate's partials are written); the next-position masks and the
// cover/uncover pass run over the particle box in one launch, whose last
// block does the step's bookkeeping. "Last block" is an atomic ticket
// per launch: no block waits for another.
#pragma once

#include "flbm_device.cuh"

namespace flbm {

// Philox4x32-10 with the round keys precomputed on the host (key + r * Weyl).
// The high and low halves of each 32 x 32-bit product are taken separately
// (this compiles to fewer instructions and registers than a 64-bit product).
__host__ __device__ __forceinline__ void philox_rk(uint32_t& x0, uint32_t& x1, uint32_t& x2, uint32_t& x3,
                                                   const KParams& P)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t h0 = mulhi32(0xD2511F53u, x0), l0 = 0xD2511F53u * x0;
        const uint32_t h1 = mulhi32(0xCD9E8D57u, x2), l1 = 0xCD9E8D57u * x2;
        const uint32_t y0 = h1 ^ x1 ^ P.rk0[r];
        const uint32_t y2 = h0 ^ x3 ^ P.rk1[r];
        x0 = y0;
        x1 = l1;
        x2 = y2;
        x3 = l0;
    }
}

// Two Box-Muller pairs from four Philox words (w1, w2 -> za0, za1; w3, w4 ->
// zb0, zb1) with the hardware approximations of log2, rsqrt, sin and cos:
// z0 = r cos(2 pi u2), z1 = r sin(2 pi u2) with r = sqrt(-2 ln u1); the angle
// is taken as 2 pi (u2 - 1/2) in (-pi, pi), where the approximations are
// accurate, and the signs flipped back. The flush-to-zero forms are used:
// their inputs and results here (u1 >= 2^-24, |angle| >= 2^-22, -2 ln u1 of
// about 2^-23 at least) lie far above the subnormal range, where both forms
// agree, and they skip the rescaling of subnormal inputs.
// The uniforms (one_to_two, as uniform_open) need no integer conversion, which
// shares the slow pipe of the four approximations. The rest of the arithmetic
// is packed over the two pairs.
__device__ __forceinline__ void box_muller2(uint32_t w1, uint32_t w2, uint32_t w3, uint32_t w4, float& za0, float& za1,
                                            float& zb0, float& zb1)
{
    const Pair u1 = add(Pair{one_to_two(w1), one_to_two(w3)}, splat(-kHalfBelowOne));
    Pair lg, rs, s, c;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg.x) : "f"(u1.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg.y) : "f"(u1.y));
    const Pair e = mul(lg, splat(-1.38629436112f));  // -2 ln u1 > 0
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.x) : "f"(e.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.y) : "f"(e.y));
    const Pair r = mul(e, rs);
    // 2 pi (u2 - 1/2) with u2 = ((w2 >> 9) + 1/2) 2^-23.
    constexpr float kA = (float)6.283185307179586;
    constexpr float kB = (float)(6.283185307179586 * (0.5 / 8388608.0 - 0.5));
    const Pair ang = mad(add(Pair{one_to_two(w2), one_to_two(w4)}, splat(-1.0f)), splat(kA), splat(kB));
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(s.x) : "f"(ang.x));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(c.x) : "f"(ang.x));
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(s.y) : "f"(ang.y));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(c.y) : "f"(ang.y));
    za0 = -r.x * c.x;
    za1 = -r.x * s.x;
    zb0 = -r.y * c.y;
    zb1 = -r.y * s.y;
}

// 1 / x and sqrt(x) from the hardware's approximations and one Newton step
// each, without the branches and calls of the general routines (__frcp_rn and
// __fsqrt_rn: 5544 -> 5715 us for 8 steps of 128x128x512 with noise). Within
// half an ulp and 2^-18 of one for 2^-126 <= x <= 2^126 and 2^-100 <= x, where
// a sweep of mantissas and exponents found CUDA's correctly rounded results
// every time; a smaller root is within 4 ulp, as its residual runs out of
// exponents. The root of zero is zero; a NaN stays one.
__device__ __forceinline__ float recip_newton(float x)
{
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}
__device__ __forceinline__ float sqrt_newton(float x)
{
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(fmaxf(x, 1.401298464e-45f)));  // the least float: a finite y for zero
    const float s = __fmul_rn(x, y);
    return __fmaf_rn(__fmaf_rn(-s, s, x), __fmul_rn(0.5f, y), s);
}

// Sums over the particle links of one node. A link exchanges m c_i, m about
// 2 w_i rho_tot; summed as they are in FP32, these cost the particle's force
// more than the rounding of the populations does, although their uniform part
// cancels around the sphere. So F holds what exceeds 2 w_i rho_l of each
// component, and k = sum 36 w_i c_i, small whole numbers, the rest, which is
// added in FP64. (The force acts along the lever c_i / 2 from the node: no
// torque about it.)
struct LinkSums {
    float F[3] = {0.0f, 0.0f, 0.0f};    // force on the particle beyond 2 w_i rho_tot c_i
    int k[3] = {0, 0, 0};
    float led[2] = {0.0f, 0.0f};        // mass put in by the moving link rule
};

// Densities and momenta of both components from their populations.
__host__ __device__ __forceinline__ void moments(const Pair f[19], Pair& rho, Pair j[3])
{
    const Pair s1 = add(f[1], f[2]), s2 = add(f[3], f[4]), s3 = add(f[5], f[6]);
    const Pair s7 = add(f[7], f[8]), s9 = add(f[9], f[10]), s11 = add(f[11], f[12]);
    const Pair s13 = add(f[13], f[14]), s15 = add(f[15], f[16]), s17 = add(f[17], f[18]);
    const Pair d7 = sub(f[7], f[8]), d9 = sub(f[9], f[10]), d11 = sub(f[11], f[12]);
    const Pair d13 = sub(f[13], f[14]), d15 = sub(f[15], f[16]), d17 = sub(f[17], f[18]);
    const Pair sax = add(add(s1, s2), s3);
    const Pair sdg = add(add(add(s7, s9), add(s11, s13)), add(s15, s17));
    rho = add(add(f[0], sax), sdg);
    j[0] = add(sub(f[1], f[2]), add(add(d7, d9), add(d11, d13)));
    j[1] = add(sub(f[3], f[4]), add(sub(d7, d9), add(d15, d17)));
    j[2] = add(sub(f[5], f[6]), add(sub(d11, d13), sub(d15, d17)));
}

// The float `bytes` beyond a base that is the same for the whole grid: a
// 32-bit offset per thread, so that the address needs no 64-bit arithmetic
// (which shares the pipe of the generator's products). A population has
// fewer than 2^32 / 38 nodes and a padded field fewer than 2^30.
__device__ __forceinline__ const float* at(const float* base, uint32_t bytes)
{
    return reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + bytes);
}
__device__ __forceinline__ float* at(float* base, uint32_t bytes)
{
    return reinterpret_cast<float*>(reinterpret_cast<char*>(base) + bytes);
}

// Where collide_core reads a node's inputs: f(i) is population i of both
// components, psi(i) the densities of neighbour x + c_i in the padded psi
// field with the components exchanged (x: rho_B, y: rho_A), as the Shan-Chen
// force of each component takes the other's.
struct GlobalInputs {
    const float* __restrict__ fin;   // current populations; (l, i) of node m at m + P.dirN[19 l + i]
    const float* __restrict__ psiA;  // padded fields of rho_A and rho_B
    const float* __restrict__ psiB;
    uint32_t n, p;                   // byte offsets of the node in a population and in a padded field
    uint32_t sy, sz;                 // padded row and plane strides in bytes
    __device__ __forceinline__ GlobalInputs(const float* f, const float* psi, int x, int y, int z, uint32_t node,
                                            const KParams& P)
        : fin(f), psiA(psi), psiB(psi + P.padn), n(4u * node),
          p(4u * ((uint32_t)(x + 1) + (uint32_t)P.px * ((uint32_t)(y + 1) + (uint32_t)P.py * (uint32_t)(z + 1)))),
          sy(4u * (uint32_t)P.px), sz(4u * (uint32_t)P.px * (uint32_t)P.py)
    {
    }
    __device__ __forceinline__ Pair f(int i, const KParams& P) const
    {
        return Pair{__ldg(at(fin + P.dirN[i], n)), __ldg(at(fin + P.dirN[19 + i], n))};
    }
    __device__ __forceinline__ Pair psi(int i) const
    {
        const uint32_t o = p + 4u * (uint32_t)cxv(i) + sy * (uint32_t)cyv(i) + sz * (uint32_t)czv(i);
        return Pair{__ldg(at(psiB, o)), __ldg(at(psiA, o))};
    }
};

// Push targets of the populations of node n = (x, y, z). Population (l, i)
// goes to the same direction's slot of node x + c_i (periodic axes wrap),
// unless c_i crosses a wall: then halfway bounce-back sends it to slot
// (l, opp(i)) of the node itself. PushFrame holds the per-node part: the
// offsets one step up and down each axis (with wrap) and which of those
// steps cross a wall.
struct PushFrame {
    int offp[3], offm[3];
    uint32_t wallp = 0, wallm = 0;
    __host__ __device__ __forceinline__ PushFrame(int x, int y, int z, const KParams& P)
    {
        const int L[3] = {P.lx, P.ly, P.lz};
        const int crd[3] = {x, y, z};
        const int stride[3] = {1, P.lx, P.lx * P.ly};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            offp[a] = stride[a];
            offm[a] = -stride[a];
            if (crd[a] + 1 >= L[a]) {
                if (P.wall[a]) wallp |= 1u << a;
                else offp[a] = stride[a] * (1 - L[a]);
            }
            if (crd[a] - 1 < 0) {
                if (P.wall[a]) wallm |= 1u << a;
                else offm[a] = stride[a] * (L[a] - 1);
            }
        }
    }
    // First direction of the pair of opposite directions i belongs to
    // (directions 2 k - 1 and 2 k; the rest direction alone).
    static __host__ __device__ constexpr int pair_of(int i) { return i == 0 || (i & 1) ? i : i - 1; }
    // Target of population i as a byte offset from slot pair_of(i) of either
    // component, and whether a wall bounced it: both candidate offsets, then
    // a select (no branch).
    __host__ __device__ __forceinline__ uint32_t target_bytes(uint32_t n, int i, const KParams& P, bool& wall) const
    {
        const int cx = cxv(i), cy = cyv(i), cz = czv(i);
        const uint32_t need_p = (cx > 0 ? 1u : 0u) | (cy > 0 ? 2u : 0u) | (cz > 0 ? 4u : 0u);
        const uint32_t need_m = (cx < 0 ? 1u : 0u) | (cy < 0 ? 2u : 0u) | (cz < 0 ? 4u : 0u);
        wall = ((wallp & need_p) | (wallm & need_m)) != 0u;
        const uint32_t N = P.dirN[1];
        int off = 0;
        if (cx) off += cx > 0 ? offp[0] : offm[0];
        if (cy) off += cy > 0 ? offp[1] : offm[1];
        if (cz) off += cz > 0 ? offp[2] : offm[2];
        const bool second = pair_of(i) != i;
        const uint32_t push = n + (uint32_t)off + (second ? N : 0u);
        const uint32_t back = n + (i != 0 && !second ? N : 0u);
        return 4u * (wall ? back : push);
    }
    // The same target as an index into the populations of component l.
    __host__ __device__ __forceinline__ uint32_t target(uint32_t n, int l, int i, const KParams& P, bool& wall) const
    {
        return P.dirN[19 * l + pair_of(i)] + target_bytes(n, i, P, wall) / 4u;
    }
};

// Receiver of the pushed populations for callers that also want the next
// step's densities (the fused bulk collide); put(i, v, bounced) sees every
// pair of populations v = f*_li the node pushes outside the particle, bounced = true
// when a wall sent it back into the node itself. The default receiver does
// nothing and compiles away.
struct NoSink {
    static constexpr bool active = false;
    __device__ __forceinline__ void put(int, Pair, bool) {}
};

// sqrt(1 / b_k): the noise amplitude of normalised mode k >= 4 per
// sqrt(3 kT rho_l) when its relaxation time is 1.
__host__ __device__ constexpr float noise_unit(int k)
{
    return k == 4 ? 1.22474487139158905f      // b = 2/3
           : k == 5 ? 0.866025403784438647f   // 4/3
           : k == 6 ? 1.5f                    // 4/9
           : k <= 9 ? 3.0f                    // 1/9
           : k <= 12 ? 1.22474487139158905f   // 2/3
           : k <= 15 ? 2.12132034355964257f   // 2/9
           : k == 16 ? 0.707106781186547524f  // 2
           : k == 17 ? 0.866025403784438647f  // 4/3
                     : 1.5f;                  // 4/9
}

// Adds the thermal noise of a node to its normalised modes n (Eq. (lbe)):
// per component variance 3 kT rho_l (1 - gamma_k^2) / b_k on mode k >= 4, and
// an interdiffusion momentum. 33 normals from 9 Philox blocks with counter
// (step, node, block, 0): A modes 4..18, B modes 4..18, interdiffusion J_x,
// J_y, J_z. Normals 2p and 2p + 1 come from Box-Muller pair p, pairs 2b and
// 2b + 1 from block b. B's mode k takes normal k + 11, the second of a pair
// where A's is the first, so the pairs are formed two at a time, p with
// p + 8, and B's odd one is kept for the next mode; modes of A and B are then
// updated together.
template <bool TAU1>
__device__ __forceinline__ void add_noise(Pair n[19], Pair rho, float irt, uint32_t node, uint32_t step,
                                          const KParams& P)
{
    const float kt3 = __fmul_rn(3.0f, P.kT);
    const float rA = fmaxf(rho.x, 0.0f), rB = fmaxf(rho.y, 0.0f);
    const Pair amp{sqrt_newton(__fmul_rn(kt3, rA)), sqrt_newton(__fmul_rn(kt3, rB))};
    auto block = [&](int b, uint32_t w[4]) {
        w[0] = step;
        w[1] = node;
        w[2] = (uint32_t)b;
        w[3] = 0u;
        philox_rk(w[0], w[1], w[2], w[3], P);
    };
    auto mode = [&](int k, float za, float zb) {
        n[k] = mad(mul(amp, splat(TAU1 ? noise_unit(k) : P.nz_mode[k])), Pair{za, zb}, n[k]);
    };
    uint32_t wa[4], wb[4];
    float z12, z13, z14, left;  // normals 12..14 (A modes 16..18) and 15 (B mode 4)
    block(3, wa);
    box_muller2(wa[0], wa[1], wa[2], wa[3], z12, z13, z14, left);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        block(b, wa);
        block(b + 4, wb);
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
            float a0, a1, b0, b1;
            box_muller2(wa[h], wa[h + 1], wb[h], wb[h + 1], a0, a1, b0, b1);
            mode(4 + 4 * b + h, a0, left);
            mode(5 + 4 * b + h, a1, b0);
            left = b1;
        }
    }
    float b0, b1, jx, jy, jz, spare;
    block(7, wa);
    block(8, wb);
    box_muller2(wa[0], wa[1], wa[2], wa[3], b0, b1, jx, jy);
    mode(16, z12, left);
    mode(17, z13, b0);
    mode(18, z14, b1);
    box_muller2(wb[0], wb[1], wb[0], wb[1], jz, spare, jz, spare);
    const float sJ =
        __fmul_rn(3.0f * P.nz_j, sqrt_newton(__fmul_rn(__fmul_rn(__fmul_rn(P.kT, rA), rB), fmaxf(irt, 0.0f))));
    const Pair pm{sJ, -sJ};
    n[1] = mad(pm, splat(jx), n[1]);
    n[2] = mad(pm, splat(jy), n[2]);
    n[3] = mad(pm, splat(jz), n[3]);
}

// What a node's update takes from its inputs: m the modes of both components
// (only rho_l and j_l, m[0..3], when every relaxation time is 1), g per axis
// the Shan-Chen sum 36 sum_i w_i c_i psi(x + c_i) (Eq. (sc-force), omega_i =
// w_i, psi = rho), the other component's densities for each.
template <bool TAU1>
struct NodeState {
    Pair m[TAU1 ? 4 : 19];
    Pair g[3];
};

template <bool TAU1, class In>
__device__ __forceinline__ void load_modes(const In& in, const KParams& P, NodeState<TAU1>& s)
{
    Pair f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = in.f(i, P);
    if constexpr (TAU1) moments(f, s.m[0], s.m + 1);
    else to_modes(f, s.m);
}

// Differences of opposite neighbours first: they are close in value.
template <bool TAU1, class In>
__host__ __device__ __forceinline__ void load_force(const In& in, NodeState<TAU1>& s)
{
    const Pair d1 = sub(in.psi(1), in.psi(2)), d2 = sub(in.psi(3), in.psi(4)), d3 = sub(in.psi(5), in.psi(6));
    const Pair d7 = sub(in.psi(7), in.psi(8)), d9 = sub(in.psi(9), in.psi(10));
    const Pair d11 = sub(in.psi(11), in.psi(12)), d13 = sub(in.psi(13), in.psi(14));
    const Pair d15 = sub(in.psi(15), in.psi(16)), d17 = sub(in.psi(17), in.psi(18));
    const Pair two = splat(2.0f);
    s.g[0] = mad(two, d1, add(add(d7, d9), add(d11, d13)));
    s.g[1] = mad(two, d2, add(sub(d7, d9), add(d15, d17)));
    s.g[2] = mad(two, d3, add(sub(d11, d13), sub(d15, d17)));
}

// Collision and push-streaming of one fluid node (Eq. (lbe)) from its loaded
// state. With PARTICLE, solid_nb marks the directions whose neighbour is a
// particle node; their links take the moving rule and give acc = (F[3], T[3],
// ledger[2]). TAU1: every relaxation time is 1, so the post-collision modes
// depend on the input only through rho_l and j_l, and the ghost modes carry
// noise only. The outputs are pushed to fout, population (l, i) of node m at
// m + P.dirN[19 l + i]. Both components go through packed arithmetic
// (flbm_pair.h).
template <bool NOISE, bool PARTICLE, bool TAU1, class In, class Sink = NoSink>
__device__ __forceinline__ void collide_push(int x, int y, int z, uint32_t n, const In& in, const NodeState<TAU1>& s,
                                             float* __restrict__ fout, const DevState* __restrict__ st,
                                             const KParams& P, uint32_t solid_nb, double* acc,
                                             Sink* sink = nullptr)
{
    const Pair* m = s.m;
    const Pair rho = m[0];
    const float irt = recip_newton(__fadd_rn(rho.x, rho.y));

    // Each component's force from the other's densities, and the external
    // force density split by rho_l.
    Pair F[3], hF[3];
    {
        const Pair gr = mul(splat(__fmul_rn(-P.G, 1.0f / 36.0f)), rho);
        const Pair share = mul(rho, splat(irt));
        const float ez = P.counterforce ? __fadd_rn(P.ext[2], st->fc_f) : P.ext[2];
        F[0] = mad(gr, s.g[0], mul(share, splat(P.ext[0])));
        F[1] = mad(gr, s.g[1], mul(share, splat(P.ext[1])));
        F[2] = mad(gr, s.g[2], mul(share, splat(ez)));
    }
    // Hydrodynamical velocity v^(H) = (sum_l j_l + (F_A + F_B)/2) / rho_tot.
    float u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        hF[a] = mul(F[a], splat(0.5f));
        const Pair jh = add(m[1 + a], hF[a]);
        u[a] = __fmul_rn(__fadd_rn(jh.x, jh.y), irt);
    }

    // MRT relaxation of both components in moment space. J = rho_l u + F_l / 2
    // is the relaxed momentum and T_ab = u_a J_b + u_b F_a / 2 the second
    // moment of equilibrium plus source.
    Pair fo[19];
    {
        Pair J[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) J[a] = mad(rho, splat(u[a]), hF[a]);
        const Pair mass = add(rho, Pair{st->delta_f[0], st->delta_f[1]});
        auto T = [&](int a, int b) { return mad(splat(u[a]), J[b], mul(splat(u[b]), hF[a])); };
        Pair k[19];  // normalised modes m_k / b_k
        k[0] = mass;
        if constexpr (TAU1) {
#pragma unroll
            for (int a = 0; a < 3; ++a) k[1 + a] = mul(J[a], splat(3.0f));
            const Pair xx = T(0, 0), yy = T(1, 1), zz = T(2, 2);
            const Pair yz = add(yy, zz), tr = add(xx, yz);
            k[4] = mul(tr, splat(1.5f));
            k[5] = mad(xx, splat(1.5f), mul(yz, splat(-0.75f)));
            k[6] = mul(sub(yy, zz), splat(2.25f));
            k[7] = mul(T(0, 1), splat(9.0f));
            k[8] = mul(T(1, 2), splat(9.0f));
            k[9] = mul(T(0, 2), splat(9.0f));
#pragma unroll
            for (int q = 10; q < 19; ++q) k[q] = splat(0.0f);
        } else {
            // equilibrium and source apart: m_eq + gamma (m - m_eq), and
            // the source by its (1 + gamma_s) / 2
            const Pair gs = splat(P.gs), gd = splat(P.gd), gg = splat(P.gg);
            const Pair h = splat(__fmul_rn(0.5f, __fadd_rn(1.0f, P.gs)));
            Pair ru[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                ru[a] = mul(rho, splat(u[a]));
                const Pair dev = sub(add(m[1 + a], hF[a]), ru[a]);
                k[1 + a] = mul(mad(gd, dev, J[a]), splat(3.0f));
            }
            Pair eq[6], S[6];
            auto eqab = [&](int a, int b) { return mul(ru[a], splat(u[b])); };
            auto sab = [&](int a, int b) { return mad(splat(u[a]), F[b], mul(splat(u[b]), F[a])); };
            const Pair exx = eqab(0, 0), eyy = eqab(1, 1), ezz = eqab(2, 2);
            const Pair sxx = sab(0, 0), syy = sab(1, 1), szz = sab(2, 2);
            const Pair eyz = add(eyy, ezz), syz = add(syy, szz);
            const Pair two = splat(2.0f);
            eq[0] = add(exx, eyz); S[0] = add(sxx, syz);
            eq[1] = sub(mul(two, exx), eyz); S[1] = sub(mul(two, sxx), syz);
            eq[2] = sub(eyy, ezz); S[2] = sub(syy, szz);
            eq[3] = eqab(0, 1); S[3] = sab(0, 1);
            eq[4] = eqab(1, 2); S[4] = sab(1, 2);
            eq[5] = eqab(0, 2); S[5] = sab(0, 2);
#pragma unroll
            for (int q = 0; q < 6; ++q)
                k[4 + q] = mul(mad(h, S[q], mad(gs, sub(m[4 + q], eq[q]), eq[q])), splat(1.0f / bnorm(4 + q)));
#pragma unroll
            for (int q = 10; q < 19; ++q) k[q] = mul(mul(gg, m[q]), splat(1.0f / bnorm(q)));
        }
        if (NOISE) add_noise<TAU1>(k, rho, irt, n, st->step_u32, P);
        from_modes(k, fo);
    }

    // Particle links of this node: sums of force and mass ledger, moved into
    // the FP64 accumulators once per node; relative position of the node to
    // the particle centre in FP64.
    LinkSums lk;
    double rn[3] = {0.0, 0.0, 0.0};
    float rnf[3] = {0.0f, 0.0f, 0.0f};
    if (PARTICLE && solid_nb) {
        rn[0] = rel_axis((double)x, st->X[0], P.lx, P.wall[0]);
        rn[1] = rel_axis((double)y, st->X[1], P.ly, P.wall[1]);
        rn[2] = rel_axis((double)z, st->X[2], P.lz, P.wall[2]);
#pragma unroll
        for (int a = 0; a < 3; ++a) rnf[a] = (float)rn[a];
    }

    // Push both components (Eq. (lbe) streaming; halfway bounce-back at
    // walls; moving link rule at the particle): the same target in each
    // component's block of populations.
    const PushFrame frame(x, y, z, P);
    float* __restrict__ foutB = fout + P.dirN[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int cx = cxv(i), cy = cyv(i), cz = czv(i);
        if (PARTICLE && (solid_nb >> i & 1u)) {
            // f_{-i}(x, t+1) = f*_i(x) - 6 w_i rho_l (u_b . c_i), u_b at the
            // link midpoint; the particle takes the momentum both exchange
            // and the reaction to the pair force with its virtual layer.
            const uint32_t back_idx = n + P.dirN[oppv(i)];
            const float r[3] = {rnf[0] + 0.5f * cx, rnf[1] + 0.5f * cy, rnf[2] + 0.5f * cz};
            const float* V = st->Vf;
            const float* Om = st->Omf;
            const float ubc = (V[0] + Om[1] * r[2] - Om[2] * r[1]) * cx + (V[1] + Om[2] * r[0] - Om[0] * r[2]) * cy +
                              (V[2] + Om[0] * r[1] - Om[1] * r[0]) * cz;
            const Pair corr = mul(rho, splat(6.0f * wv(i) * ubc));
            const Pair back = sub(fo[i], corr);
            fout[back_idx] = back.x;
            foutB[back_idx] = back.y;
            const Pair pn = in.psi(i), mw = splat(-wv(i));
            const Pair ex = add(mad(mw, rho, fo[i]), mad(mw, rho, back));
            const float m = (ex.x + ex.y) + P.G * wv(i) * (rho.x * pn.x + rho.y * pn.y);
            lk.F[0] += m * cx; lk.F[1] += m * cy; lk.F[2] += m * cz;
            const int w36 = i <= 6 ? 2 : 1;
            lk.k[0] += w36 * cx; lk.k[1] += w36 * cy; lk.k[2] += w36 * cz;
            lk.led[0] += corr.x;
            lk.led[1] += corr.y;
            continue;
        }
        bool wall;
        const uint32_t to = frame.target_bytes(n, i, P, wall);
        const int pair = PushFrame::pair_of(i);
        *at(fout + P.dirN[pair], to) = fo[i].x;
        *at(fout + P.dirN[19 + pair], to) = fo[i].y;
        if constexpr (Sink::active) sink->put(i, fo[i], wall);
    }
    if (PARTICLE && solid_nb) {
        const double base = 2.0 * (double)wv(7) * ((double)rho.x + (double)rho.y);
        double F[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) F[a] = (double)lk.F[a] + base * (double)lk.k[a];
        acc[0] = F[0]; acc[1] = F[1]; acc[2] = F[2];
        acc[3] = rn[1] * F[2] - rn[2] * F[1];
        acc[4] = rn[2] * F[0] - rn[0] * F[2];
        acc[5] = rn[0] * F[1] - rn[1] * F[0];
        acc[6] = lk.led[0];
        acc[7] = lk.led[1];
    }
}

// The whole update of a node from one set of inputs.
template <bool NOISE, bool PARTICLE, bool TAU1, class In, class Sink = NoSink>
__device__ __forceinline__ void collide_core(int x, int y, int z, uint32_t n, const In& in,
                                             float* __restrict__ fout, const DevState* __restrict__ st,
                                             const KParams& P, uint32_t solid_nb, double* acc,
                                             Sink* sink = nullptr)
{
    NodeState<TAU1> s;
    load_modes(in, P, s);
    load_force(in, s);
    collide_push<NOISE, PARTICLE, TAU1>(x, y, z, n, in, s, fout, st, P, solid_nb, acc, sink);
}

// collide_core with its inputs read from global memory.
template <bool NOISE, bool PARTICLE, bool TAU1>
__device__ __forceinline__ void collide_node(int x, int y, int z, uint32_t n, const float* __restrict__ fin,
                                             float* __restrict__ fout, const float* __restrict__ psi,
                                             const DevState* __restrict__ st, const KParams& P, uint32_t solid_nb,
                                             double* acc)
{
    const GlobalInputs in(fin, psi, x, y, z, n, P);
    collide_core<NOISE, PARTICLE, TAU1>(x, y, z, n, in, fout, st, P, solid_nb, acc);
}

// ---------------------------------------------------------------------------
// Bulk tiles: every tile not next to the particle.
// ---------------------------------------------------------------------------
// Thread (tx, ty) of tile (bx, by, bz).
template <bool NOISE, bool TAU1>
__device__ __forceinline__ void bulk_tile(int bx, int by, int bz, int tx, int ty, const float* __restrict__ fin,
                                          float* __restrict__ fout, const float* __restrict__ psi,
                                          const DevState* __restrict__ st, const KParams& P)
{
    if (P.has_particle) {
        const int o[3] = {st->box0[0], st->box0[1], st->box0[2]};
        if (tile_near(bx, by, bz, o, P)) return;
    }
    const int x = bx * P.tx + tx;
    const int y = by * P.ty + ty;
    const int z = bz;
    if (x >= P.lx || y >= P.ly) return;
    const uint32_t n = (uint32_t)x + (uint32_t)P.lx * ((uint32_t)y + (uint32_t)P.ly * (uint32_t)z);
    collide_node<NOISE, false, TAU1>(x, y, z, n, fin, fout, psi, st, P, 0u, nullptr);
}

// Blocks of the bulk launches: part (0 .. kBulkParts - 1) of a tile, its rows
// ty / kBulkParts * part onwards. With noise two blocks of 128 threads share
// a tile, seven per SM: 72 registers hold the update without spills (a
// spilled register's store goes through to L2), and a half block's slot is
// refilled sooner. Collide of 128x128x512: 459 us, against 478 us for whole
// tiles at four blocks of 64 registers and 530 us at three of 80. Without
// noise 64 registers suffice and the four whole tiles are best: 432 us
// against 447 us.
template <bool NOISE>
constexpr int kBulkParts = NOISE ? 2 : 1;
template <bool NOISE>
constexpr int kBulkThreads = kThreadsStep / kBulkParts<NOISE>;
template <bool NOISE>
constexpr int kBulkBlocks = NOISE ? 7 : 4;  // resident per SM

template <bool NOISE, bool TAU1>
static __global__ void __launch_bounds__(kBulkThreads<NOISE>, kBulkBlocks<NOISE>)
    k_collide_bulk(const float* __restrict__ fin, float* __restrict__ fout, const float* __restrict__ psi,
                   const DevState* __restrict__ st, KParams P)
{
    constexpr unsigned parts = kBulkParts<NOISE>;
    bulk_tile<NOISE, TAU1>(blockIdx.x / parts, blockIdx.y, blockIdx.z, threadIdx.x,
                           threadIdx.y + blockDim.y * (blockIdx.x % parts), fin, fout, psi, st, P);
}

// Candidate c on one axis -> tile index, or -1. e0 = first coordinate of the
// grown box on that axis; tiles of size T, gt of them, axis length L.
__host__ __device__ __forceinline__ int candidate_tile(int c, int o, int T, int gt, int L, int wall)
{
    int e0 = o - 1;
    if (wall) {
        if (e0 < 0) e0 = 0;
        const int t = e0 / T + c;
        return t < gt ? t : -1;
    }
    if (e0 < 0) e0 += L;
    return (e0 / T + c) % gt;
}

// ---------------------------------------------------------------------------
// Near tiles: a fixed grid of candidate tiles around the particle box; each
// near tile reduces force, torque and mass ledger into partials[candidate].
// ---------------------------------------------------------------------------
// Candidate (cx, cy, cz) of the grid around the particle box; thread (tx, ty)
// of the tile, tid = tx + TX ty. Every thread of the block must call this.
template <bool NOISE, bool TAU1>
__device__ __forceinline__ void near_tile_work(int cx, int cy, int cz, int tx, int ty, int tid,
                                          const float* __restrict__ fin, float* __restrict__ fout,
                                          const float* __restrict__ psi, const DevState* __restrict__ st,
                                          const uint8_t* __restrict__ masks, double* __restrict__ partials,
                                          const KParams& P)
{
    __shared__ double s_red[(kThreadsStep / 32) * 8];
    __shared__ double s_out[8];
    const int o[3] = {st->box0[0], st->box0[1], st->box0[2]};
    const int bx = candidate_tile(cx, o[0], P.tx, P.gx, P.lx, P.wall[0]);
    const int by = candidate_tile(cy, o[1], P.ty, P.gy, P.ly, P.wall[1]);
    const int bz = candidate_tile(cz, o[2], 1, P.lz, P.lz, P.wall[2]);
    const long long cand = cx + (long long)P.ncx * (cy + (long long)P.ncy * cz);
    const bool near = bx >= 0 && by >= 0 && bz >= 0 && tile_near(bx, by, bz, o, P);
    if (!near) {
        if (tid < 8) partials[cand * 8 + tid] = 0.0;
        return;
    }
    const uint8_t* mask = masks + (size_t)st->cur * P.B * P.B * P.B;
    const int x = bx * P.tx + tx;
    const int y = by * P.ty + ty;
    const int z = bz;
    const bool inside = x < P.lx && y < P.ly;
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const bool fluid = inside && !is_solid(x, y, z, o, mask, P);
    const uint32_t links = fluid ? solid_neighbours(x, y, z, o, mask, P) : 0u;
    // A warp none of whose nodes has a particle link takes the update of the
    // bulk tiles. Every lane of the block's full warps reaches the vote.
    const bool warp_links = __any_sync(0xffffffffu, links != 0u);
    if (fluid) {
        const uint32_t n = (uint32_t)x + (uint32_t)P.lx * ((uint32_t)y + (uint32_t)P.ly * (uint32_t)z);
        if (warp_links) collide_node<NOISE, true, TAU1>(x, y, z, n, fin, fout, psi, st, P, links, acc);
        else collide_node<NOISE, false, TAU1>(x, y, z, n, fin, fout, psi, st, P, 0u, nullptr);
    }
    if (!__syncthreads_or(links != 0)) {  // no particle link in this tile
        if (tid < 8) partials[cand * 8 + tid] = 0.0;
        return;
    }
    block_sum8<kThreadsStep>(acc, s_red, s_out, links != 0);
    if (tid < 8) partials[cand * 8 + tid] = s_out[tid];
    __syncthreads();  // s_out is reused by the next tile of a persistent block
}

__device__ __forceinline__ void update_particle(DevState* __restrict__ st, const double* __restrict__ partials,
                                                const KParams& P);

// A near tile, then, in the block that finishes the launch's last candidate,
// the particle update of this step (sum of all candidates' partials in fixed
// order, leap-frog).
template <bool NOISE, bool TAU1>
__device__ __forceinline__ void near_tile(int cx, int cy, int cz, int tx, int ty, int tid,
                                          const float* __restrict__ fin, float* __restrict__ fout,
                                          const float* __restrict__ psi, DevState* __restrict__ st,
                                          const uint8_t* __restrict__ masks, double* __restrict__ partials,
                                          const KParams& P)
{
    near_tile_work<NOISE, TAU1>(cx, cy, cz, tx, ty, tid, fin, fout, psi, st, masks, partials, P);
    if (last_block(&st->near_done, (unsigned)(P.ncx * P.ncy * P.ncz), tid < 8))  // tid < 8 wrote partials
        update_particle(st, partials, P);
    __syncthreads();
}

// Two blocks per SM (128 registers): the links' code beside the bulk update
// spills at three (collide class of 64x64x128: 37.5 us against 51.5 us).
template <bool NOISE, bool TAU1>
static __global__ void __launch_bounds__(kThreadsStep, 2)
    k_collide_near(const float* __restrict__ fin, float* __restrict__ fout, const float* __restrict__ psi,
                   DevState* __restrict__ st, const uint8_t* __restrict__ masks,
                   double* __restrict__ partials, KParams P)
{
    near_tile<NOISE, TAU1>(blockIdx.x, blockIdx.y, blockIdx.z, threadIdx.x, threadIdx.y,
                           threadIdx.x + blockDim.x * threadIdx.y, fin, fout, psi, st, masks, partials, P);
}

__host__ __device__ __forceinline__ void box_origin(const double X[3], const KParams& P, int o[3])
{
    const int L[3] = {P.lx, P.ly, P.lz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = (int)floor(X[a] - P.R);
        if (!P.wall[a]) {
            v %= L[a];
            if (v < 0) v += L[a];
        }
        o[a] = v;
    }
}

// Is lattice node c strictly inside the sphere around X (FP64)?
__host__ __device__ __forceinline__ bool node_inside(const int c[3], const double X[3], const KParams& P)
{
    const int L[3] = {P.lx, P.ly, P.lz};
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double r = rel_axis((double)c[a], X[a], L[a], P.wall[a]);
        s += r * r;
    }
    return s < P.R * P.R;
}

// Particle node test for box entry t of a box at origin o around centre X (FP64).
__host__ __device__ __forceinline__ bool box_node_inside(int t, const int o[3], const double X[3], const KParams& P)
{
    const int B = P.B;
    const int d[3] = {t % B, (t / B) % B, t / (B * B)};
    const int L[3] = {P.lx, P.ly, P.lz};
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c[a] = o[a] + d[a];
        if (P.wall[a]) {
            if (c[a] < 0 || c[a] >= L[a]) return false;
        } else if (c[a] >= L[a]) {
            c[a] -= L[a];
        }
    }
    return node_inside(c, X, P);
}

// ---------------------------------------------------------------------------
// (1) Sum the near-tile partials in candidate order, leap-frog update (FP64),
// new box origin. One block.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void update_particle(DevState* __restrict__ st, const double* __restrict__ partials,
                                                const KParams& P)
{
    __shared__ double s_red[(256 / 32) * 8];
    __shared__ double s_out[8];
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    // The record's values are loaded before the sum, which their latency then
    // overlaps.
    const int a = tid;
    double Pp = 0.0, Lp = 0.0, v0 = 0.0, om0 = 0.0, x0 = 0.0, ext = 0.0;
    if (a < 3) {
        Pp = st->Ppend[a];
        Lp = st->Lpend[a];
        v0 = st->V[a];
        om0 = st->Om[a];
        x0 = st->X[a];
        ext = (a == 2) ? st->Fp : 0.0;
    }
    sum_rows8(partials, (long long)P.ncx * P.ncy * P.ncz, s_red, s_out);
    // One thread per axis: the three components are independent. FP64 on a
    // part whose FP64 is slow, so products with 1 / m_p and 1 / I_p, and the
    // periodic wrap as a conditional shift (floor only for a longer step).
    if (a >= 3) return;
    const int L = a == 0 ? P.lx : (a == 1 ? P.ly : P.lz);
    const double F = s_out[a] + Pp;
    const double T = s_out[3 + a] + Lp;
    st->F[a] = F;
    st->T[a] = T;
    const double vn = v0 + (F + ext) * P.inv_mp;
    st->Vavg[a] = 0.5 * (v0 + vn);
    st->V[a] = vn;
    const double om = om0 + T * P.inv_Ip;
    st->Om[a] = om;
    st->Vf[a] = (float)vn;
    st->Omf[a] = (float)om;
    double xn = x0 + vn;
    if (!P.wall[a]) {
        if (xn >= L) xn -= L;
        else if (xn < 0.0) xn += L;
        if (xn >= L || xn < 0.0) xn -= L * floor(xn / L);
    }
    st->X[a] = xn;
    if (a == 0) {
        st->ledger_bb[0] = s_out[6];
        st->ledger_bb[1] = s_out[7];
    }
    // box_origin of the new position, this axis.
    int o = (int)floor(xn - P.R);
    if (!P.wall[a]) {
        o %= L;
        if (o < 0) o += L;
    }
    st->box_next[a] = o;
}

// Sums of the 19 populations of both components at node m, no less exact than
// in FP64, by cascaded float two-sums (Ogita, Rump and Oishi's SumK, K = 3: within
// 2^-56 of the magnitudes), so that the slow FP64 pipe only sees
// the three partial results. 16x16x32 takes 502 us for 16 steps, 517 us with
// the 38 conversions and additions of a lane in FP64.
__host__ __device__ __forceinline__ void pop_sums(const float* __restrict__ f, long long m, long long N, double r[2])
{
    Pair v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = Pair{f[(long long)i * N + m], f[(long long)(19 + i) * N + m]};
    Pair s = v[0], t = splat(0.0f), g = splat(0.0f);
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        Pair e, h;
        two_sum(s, v[i], s, e);
        two_sum(t, e, t, h);
        g = add(g, h);
    }
    r[0] = (double)s.x + ((double)t.x + (double)g.x);
    r[1] = (double)s.y + ((double)t.y + (double)g.y);
}

// c_i along axis a for a direction known at run time: +1, 0 or -1.
__device__ __forceinline__ int dir_of(int i, int a)
{
    constexpr uint32_t p[3] = {1u << 1 | 1u << 7 | 1u << 9 | 1u << 11 | 1u << 13,
                               1u << 3 | 1u << 7 | 1u << 10 | 1u << 15 | 1u << 17,
                               1u << 5 | 1u << 11 | 1u << 14 | 1u << 15 | 1u << 18};
    constexpr uint32_t m[3] = {1u << 2 | 1u << 8 | 1u << 10 | 1u << 12 | 1u << 14,
                               1u << 4 | 1u << 8 | 1u << 9 | 1u << 16 | 1u << 18,
                               1u << 6 | 1u << 12 | 1u << 13 | 1u << 16 | 1u << 17};
    const uint32_t pa = a == 0 ? p[0] : (a == 1 ? p[1] : p[2]), ma = a == 0 ? m[0] : (a == 1 ? m[1] : m[2]);
    return (int)(pa >> i & 1u) - (int)(ma >> i & 1u);
}
__device__ __forceinline__ double signed_by(int s, double v) { return s == 0 ? 0.0 : (s > 0 ? v : -v); }

// Component k of (p, r x p, mass): lane k's share of what an event at r gives.
__device__ __forceinline__ double event_value(int k, const double r[3], const double p[3], double mA, double mB)
{
    const int a = k >= 3 ? k - 3 : k;
    const double rb = a == 0 ? r[1] : (a == 1 ? r[2] : r[0]), rc = a == 0 ? r[2] : (a == 1 ? r[0] : r[1]);
    const double pb = a == 0 ? p[1] : (a == 1 ? p[2] : p[0]), pc = a == 0 ? p[2] : (a == 1 ? p[0] : p[1]);
    const double cross = rb * pc - rc * pb;
    const double lin = k == 0 ? p[0] : (k == 1 ? p[1] : p[2]);
    return k < 3 ? lin : (k < 6 ? cross : (k == 6 ? mA : mB));
}

// node_inside decided in float where the distance is clear of the surface by
// more than the float's error can reach (coordinates good to 2^-23 of the
// longest axis, squared distances within the box and its neighbours to that
// times 4 (R + 4) and a few ulps), else in FP64: few nodes need the slow pipe.
struct SphereTest {
    float x[3], R2, margin;
    __host__ __device__ __forceinline__ SphereTest(const double X[3], const KParams& P)
    {
        const float R = (float)P.R;
#pragma unroll
        for (int a = 0; a < 3; ++a) x[a] = (float)X[a];
        R2 = R * R;
        margin = 1e-6f * ((R + 4.0f) * (float)max(P.lx, max(P.ly, P.lz)) + 8.0f * R2) + 1e-5f;
    }
    __host__ __device__ __forceinline__ bool inside(const int c[3], const double X[3], const KParams& P) const
    {
        const int L[3] = {P.lx, P.ly, P.lz};
        float s = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float r = (float)c[a] - x[a];
            if (!P.wall[a]) {
                if (r > 0.5f * L[a]) r -= L[a];
                else if (r < -0.5f * L[a]) r += L[a];
            }
            s += r * r;
        }
        if (fabsf(s - R2) > margin) return s < R2;
        return node_inside(c, X, P);
    }
};

// (2) Particle nodes at the new position -> mask[1 - cur] and their count,
// cover (new box) and uncover (old box) on the post-stream populations f;
// per-block FP64 partials of impulse, angular impulse and mass ledger. Block
// blk of 256 box entries. No thread reads what another marks: where a node's
// new state is asked it is tested again.
//
// The events of a warp's entries are taken one after the other by the whole
// warp: its lanes share the populations, the neighbours and the axes, and lane
// k keeps the k-th of the eight sums. One thread per event held the step's
// critical path for 8 to 10 us of chained FP64.
__device__ __forceinline__ void cover_block(int blk, float* __restrict__ f, const DevState* __restrict__ st,
                                            uint8_t* __restrict__ masks, int* __restrict__ counts,
                                            double* __restrict__ parts, const KParams& P)
{
    __shared__ double s_red[(256 / 32) * 8];
    __shared__ int s_cnt[256 / 32];
    __shared__ int s_any;
    const int B = P.B;
    const int B3 = B * B * B;
    const int t = blk * 256 + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int cur = st->cur;
    const int o_old[3] = {st->box0[0], st->box0[1], st->box0[2]};
    const int o_new[3] = {st->box_next[0], st->box_next[1], st->box_next[2]};
    const double X[3] = {st->X[0], st->X[1], st->X[2]};
    const uint8_t* m_old = masks + (size_t)cur * B3;
    const int L[3] = {P.lx, P.ly, P.lz};
    const long long N = P.N;
    const SphereTest sphere(X, P);
    if (threadIdx.x == 0) s_any = 0;
    bool now = false, covered = false, uncovered = false;
    int cc[3] = {0, 0, 0}, cu_[3] = {0, 0, 0};  // the covered / uncovered node of this thread
    if (t < B3) {
        const int d[3] = {t % B, (t / B) % B, t / (B * B)};
        const bool was = m_old[t] != 0;
        now = true;
        for (int a = 0; a < 3; ++a) {
            cc[a] = o_new[a] + d[a];
            if (P.wall[a]) now = now && cc[a] >= 0 && cc[a] < L[a];
            else if (cc[a] >= L[a]) cc[a] -= L[a];
        }
        now = now && sphere.inside(cc, X, P);
        masks[(size_t)(1 - cur) * B3 + t] = (uint8_t)now;
        if (now) covered = !is_solid(cc[0], cc[1], cc[2], o_old, m_old, P);
        if (was) {
            for (int a = 0; a < 3; ++a) {
                cu_[a] = o_old[a] + d[a];
                if (!P.wall[a] && cu_[a] >= L[a]) cu_[a] -= L[a];
            }
            uncovered = !sphere.inside(cu_, X, P);
        }
    }
    const unsigned marked = __ballot_sync(0xffffffffu, now);
    unsigned cm = __ballot_sync(0xffffffffu, covered), um = __ballot_sync(0xffffffffu, uncovered);
    double acc = 0.0;  // lanes 0..7: the warp's sum of that component
    const bool events = (cm | um) != 0u;
    // Covered nodes: lane q holds population q, lanes 0..5 also 32 + q.
    while (cm) {
        const int src = __ffs(cm) - 1;
        cm &= cm - 1;
        int c[3];
        for (int a = 0; a < 3; ++a) c[a] = __shfl_sync(0xffffffffu, cc[a], src);
        const long long n = c[0] + (long long)P.lx * (c[1] + (long long)P.ly * c[2]);
        const double f0 = f[(long long)lane * N + n];
        const double f1 = lane < 6 ? (double)f[(long long)(32 + lane) * N + n] : 0.0;
        const int i0 = lane < 19 ? lane : lane - 19, i1 = 13 + lane;
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int a = 0; a < 3; ++a)
            v[a] = signed_by(dir_of(i0, a), f0) + (lane < 6 ? signed_by(dir_of(i1, a), f1) : 0.0);
        v[3] = lane < 19 ? f0 : 0.0;
        v[4] = (lane < 19 ? 0.0 : f0) + f1;
        const double s = warp_sum8(v, lane);
        double p[3], r[3];
        double ra = 0.0;
        if (lane < 3) {
            const int ca = lane == 0 ? c[0] : (lane == 1 ? c[1] : c[2]);
            const double Xa = lane == 0 ? X[0] : (lane == 1 ? X[1] : X[2]);
            const int La = lane == 0 ? L[0] : (lane == 1 ? L[1] : L[2]);
            ra = rel_axis((double)ca, Xa, La, P.wall[lane]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            p[a] = __shfl_sync(0xffffffffu, s, sum_lane(a));
            r[a] = __shfl_sync(0xffffffffu, ra, a);
        }
        const double mA = __shfl_sync(0xffffffffu, s, sum_lane(3)), mB = __shfl_sync(0xffffffffu, s, sum_lane(4));
        acc += event_value(lane & 7, r, p, mA, mB);
    }
    // Uncovered nodes: lane j (1..18) sums the populations of neighbour j,
    // the warp adds them up (exact sums), and the lanes write the refilled
    // populations.
    while (um) {
        const int src = __ffs(um) - 1;
        um &= um - 1;
        int c[3];
        for (int a = 0; a < 3; ++a) c[a] = __shfl_sync(0xffffffffu, cu_[a], src);
        double ml[2] = {0.0, 0.0};
        bool ok = false;
        if (lane >= 1 && lane <= 18) {
            int q[3] = {c[0] + dir_of(lane, 0), c[1] + dir_of(lane, 1), c[2] + dir_of(lane, 2)};
            ok = true;
            for (int a = 0; a < 3; ++a) {
                if (q[a] < 0 || q[a] >= L[a]) {
                    if (P.wall[a]) ok = false;
                    else q[a] += (q[a] < 0) ? L[a] : -L[a];
                }
            }
            // a fluid neighbour that was fluid before as well
            ok = ok && !is_solid(q[0], q[1], q[2], o_old, m_old, P) && !sphere.inside(q, X, P);
            if (ok) {
                const long long m = q[0] + (long long)P.lx * (q[1] + (long long)P.ly * q[2]);
                pop_sums(f, m, N, ml);
            }
        }
        const int cnt = __popc(__ballot_sync(0xffffffffu, ok));
        // lanes 0..15 end with component A, lanes 16..31 with B
        const bool up = lane >= 16;
        double ms = (up ? ml[1] : ml[0]) + __shfl_xor_sync(0xffffffffu, up ? ml[0] : ml[1], 16);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) ms += __shfl_xor_sync(0xffffffffu, ms, off);
        // neighbour-mean densities; the initial densities if no fluid neighbour is left
        const double rl = cnt ? ms / cnt : (up ? P.rho0[1] : P.rho0[0]);
        const double rA = __shfl_sync(0xffffffffu, rl, 0), rB = __shfl_sync(0xffffffffu, rl, 16);
        double r[3], ub[3], ra = 0.0, ua = 0.0;
        if (lane < 3) {
            const int ca = lane == 0 ? c[0] : (lane == 1 ? c[1] : c[2]);
            const double Xa = lane == 0 ? X[0] : (lane == 1 ? X[1] : X[2]);
            const int La = lane == 0 ? L[0] : (lane == 1 ? L[1] : L[2]);
            ra = rel_axis((double)ca, Xa, La, P.wall[lane]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) r[a] = __shfl_sync(0xffffffffu, ra, a);
        if (lane < 3) {
            const int b = lane == 2 ? 0 : lane + 1, e = lane == 0 ? 2 : lane - 1;
            const double rb = b == 0 ? r[0] : (b == 1 ? r[1] : r[2]), re = e == 0 ? r[0] : (e == 1 ? r[1] : r[2]);
            ua = st->V[lane] + st->Om[b] * re - st->Om[e] * rb;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) ub[a] = __shfl_sync(0xffffffffu, ua, a);
        const long long n = c[0] + (long long)P.lx * (c[1] + (long long)P.ly * c[2]);
        const double base = 1.0 - 1.5 * (ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2]);
        for (int q = lane; q < 38; q += 32) {  // population (l, i) = (q / 19, q % 19)
            const int l = q >= 19, i = q - 19 * l;
            const double cu =
                signed_by(dir_of(i, 0), ub[0]) + signed_by(dir_of(i, 1), ub[1]) + signed_by(dir_of(i, 2), ub[2]);
            f[(long long)q * N + n] = (float)(wv(i) * (l ? rB : rA) * (base + cu * (3.0 + 4.5 * cu)));
        }
        const double rt = rA + rB;
        const double p[3] = {rt * ub[0], rt * ub[1], rt * ub[2]};
        acc -= event_value(lane & 7, r, p, rA, rB);
    }
    __syncthreads();  // s_any is cleared
    if (lane < 8) s_red[(threadIdx.x >> 5) * 8 + lane] = acc;
    if (lane == 0) {
        s_cnt[threadIdx.x >> 5] = __popc(marked);
        if (events) s_any = 1;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        double s = 0.0;
        if (s_any)
            for (int w = 0; w < 256 / 32; ++w) s += s_red[w * 8 + threadIdx.x];
        parts[blk * 8 + threadIdx.x] = s;
    }
    if (threadIdx.x == 0) {
        int a = 0;
        for (int w = 0; w < 256 / 32; ++w) a += s_cnt[w];
        counts[blk] = a;
    }
    __syncthreads();
}

__device__ __forceinline__ void finish_step(DevState* __restrict__ st, const int* __restrict__ counts,
                                            const double* __restrict__ parts, int nblocks, const KParams& P);

// A block of the cover/uncover pass, then, in the launch's last block, the
// step's bookkeeping (finish_step).
__device__ __forceinline__ void cover_then_finish(int blk, float* __restrict__ f, DevState* __restrict__ st,
                                                  uint8_t* __restrict__ masks, double* __restrict__ parts,
                                                  int* __restrict__ counts, const KParams& P)
{
    cover_block(blk, f, st, masks, counts, parts, P);
    const int nb = (P.B * P.B * P.B + 255) / 256;
    if (last_block(&st->cover_done, (unsigned)nb, threadIdx.x < 8))  // threads 0..7 wrote parts and the count
        finish_step(st, counts, parts, nb, P);
    __syncthreads();
}

static __global__ void __launch_bounds__(256) k_cover(float* __restrict__ f, DevState* __restrict__ st,
                                                      uint8_t* __restrict__ masks, double* __restrict__ parts,
                                                      int* __restrict__ counts, KParams P)
{
    cover_then_finish(blockIdx.x, f, st, masks, parts, counts, P);
}

// (4) Bookkeeping for the next step: pending impulses, fluid count, mass
// correction delta_l = ledger_l / N_fluid, counterforce, box swap, step + 1.
// Without a particle only the step counter advances. One block.
__device__ __forceinline__ void finish_step(DevState* __restrict__ st, const int* __restrict__ counts,
                                            const double* __restrict__ parts, int nblocks, const KParams& P)
{
    __shared__ double s_red[(256 / 32) * 8];
    __shared__ double s_out[8];
    __shared__ long long s_c[256 / 32];
    if (!P.has_particle) {
        if (threadIdx.x == 0) {
            st->step += 1;
            st->step_u32 = (uint32_t)st->step;
        }
        return;
    }
    // The record's values are loaded before the sums.
    double led = 0.0, Fp = 0.0;
    if (threadIdx.x < 2) led = st->ledger_bb[threadIdx.x];
    if (threadIdx.x == 2) Fp = st->Fp;
    const long long step = st->step;
    const int cur = st->cur;
    int box[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        box[a] = st->box0[a];
        box[3 + a] = st->box_next[a];
    }
    long long cnt = 0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) cnt += __ldcg(counts + b);
    // Particle nodes: an integer sum, the same in any order.
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    if ((threadIdx.x & 31) == 0) s_c[threadIdx.x >> 5] = cnt;
    sum_rows8(parts, nblocks, s_red, s_out);  // its barriers also publish s_c
    // Threads 0, 1, 2 form delta_A, delta_B and the counterforce at once
    // (FP64 divisions are slow here); thread 0 also the rest.
    if (threadIdx.x >= 3) return;
    long long solid = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) solid += s_c[w];
    const long long nf = P.N - solid;
    if (threadIdx.x < 2) {
        const int l = threadIdx.x;
        const double delta = (led + s_out[6 + l]) / (double)nf;
        st->delta[l] = delta;
        st->delta_f[l] = (float)delta;
    } else {
        const double fc = P.counterforce ? -Fp / (double)nf : 0.0;
        st->fc = fc;
        st->fc_f = (float)fc;
    }
    if (threadIdx.x != 0) return;
    for (int a = 0; a < 3; ++a) {
        st->Ppend[a] = s_out[a];
        st->Lpend[a] = s_out[3 + a];
    }
    st->nfluid = nf;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        st->box_prev[a] = box[a];
        st->box0[a] = box[3 + a];
    }
    st->cur = 1 - cur;
    st->step = step + 1;
    st->step_u32 = (uint32_t)(step + 1);
}

static __global__ void __launch_bounds__(256) k_finish(DevState* __restrict__ st, const int* __restrict__ counts,
                                                       const double* __restrict__ parts, int nblocks, KParams P)
{
    finish_step(st, counts, parts, nblocks, P);
}

// Mark the particle nodes of the current position into mask[cur] and set the
// box origin, fluid count and counterforce (creation and flbm_set_particle).
// One block; FP64 inside test as in the step.
static __global__ void __launch_bounds__(1024) k_mark(DevState* st, uint8_t* masks, KParams P)
{
    __shared__ long long s_c[1024];
    __shared__ int s_o[3];
    if (threadIdx.x == 0) {
        int o[3];
        box_origin(st->X, P, o);
        s_o[0] = o[0]; s_o[1] = o[1]; s_o[2] = o[2];
    }
    __syncthreads();
    const int o[3] = {s_o[0], s_o[1], s_o[2]};
    const double X[3] = {st->X[0], st->X[1], st->X[2]};
    const int B3 = P.B * P.B * P.B;
    uint8_t* mask = masks + (size_t)st->cur * B3;
    long long cnt = 0;
    for (int t = threadIdx.x; t < B3; t += blockDim.x) {
        const bool in = box_node_inside(t, o, X, P);
        mask[t] = in ? 1 : 0;
        cnt += in;
    }
    s_c[threadIdx.x] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long a = 0;
        for (int k = 0; k < (int)blockDim.x; ++k) a += s_c[k];
        st->box0[0] = o[0]; st->box0[1] = o[1]; st->box0[2] = o[2];
        st->nfluid = P.N - a;
        st->fc = (P.counterforce && st->nfluid > 0) ? -st->Fp / (double)st->nfluid : 0.0;
        st->fc_f = (float)st->fc;
        st->delta_f[0] = (float)st->delta[0];
        st->delta_f[1] = (float)st->delta[1];
        st->step_u32 = (uint32_t)st->step;
        for (int a = 0; a < 3; ++a) {
            st->Vf[a] = (float)st->V[a];
            st->Omf[a] = (float)st->Om[a];
        }
    }
}

}  // namespace flbm
