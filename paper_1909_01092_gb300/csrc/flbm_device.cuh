// Device code of the FLBM step: lattice, Philox, and the kernels.
//
// Method: arXiv:1909.01092, Section 2 (Eqs. (density), (lbe), (sc-force), the
// particle coupling paragraph) and Section 3 (Eq. (fp), channel walls).
//
// Data layout in HBM (N = lx*ly*lz, x fastest):
//   f[2 copies][2 components][19 directions][N]     float32, post-stream state
//   psi[2 components][lz+2][ly+2][lx+2]              float32, densities with a
//        one-node shell: copies across periodic faces, neutral wall ghosts
//        across walled faces; virtual-layer values on particle surface nodes
//   mask[2][B^3]                                     uint8, particle nodes in a
//        cube of side B around the sphere (current and next position)
//   partials[tiles][8]                               float64, per-tile force,
//        torque and mass ledger of tiles next to the particle
//   DevState                                         float64 particle state
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "flbm_pair.h"

namespace flbm {

// ---------------------------------------------------------------------------
// D3Q19 (Section 2). Direction order: rest, +-x, +-y, +-z, xy, xz, yz pairs.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int cxv(int i)
{
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ constexpr int cyv(int i)
{
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
           : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ constexpr int czv(int i)
{
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
           : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
__host__ __device__ constexpr int oppv(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
__host__ __device__ constexpr float wv(int i) { return i == 0 ? 1.0f / 3.0f : (i <= 6 ? 1.0f / 18.0f : 1.0f / 36.0f); }

// Norms b_k of the mode basis (sum_i w_i e_k(c_i)^2).
__host__ __device__ constexpr float bnorm(int k)
{
    return k == 0 ? 1.0f
           : k <= 3 ? 1.0f / 3.0f
           : k == 4 ? 2.0f / 3.0f
           : k == 5 ? 4.0f / 3.0f
           : k == 6 ? 4.0f / 9.0f
           : k <= 9 ? 1.0f / 9.0f
           : k <= 12 ? 2.0f / 3.0f
           : k <= 15 ? 2.0f / 9.0f
           : k == 16 ? 2.0f
           : k == 17 ? 4.0f / 3.0f : 4.0f / 9.0f;
}

// Forward mode transform m_k = sum_i e_k(c_i) f_i of the D3Q19 MRT basis
// (density, momentum, 6 stress, 9 ghost modes), evaluated with opposite-pair
// sums (even modes) and differences (odd modes), every operation written out;
// T = Pair in the step (both components at once), double in the observables.
template <class T>
__host__ __device__ __forceinline__ void to_modes(const T f[19], T m[19])
{
    const T two = lit<T>(2.0f), mtwo = lit<T>(-2.0f);
    const T s1 = add(f[1], f[2]), d1 = sub(f[1], f[2]);
    const T s2 = add(f[3], f[4]), d2 = sub(f[3], f[4]);
    const T s3 = add(f[5], f[6]), d3 = sub(f[5], f[6]);
    const T s7 = add(f[7], f[8]), d7 = sub(f[7], f[8]);
    const T s9 = add(f[9], f[10]), d9 = sub(f[9], f[10]);
    const T s11 = add(f[11], f[12]), d11 = sub(f[11], f[12]);
    const T s13 = add(f[13], f[14]), d13 = sub(f[13], f[14]);
    const T s15 = add(f[15], f[16]), d15 = sub(f[15], f[16]);
    const T s17 = add(f[17], f[18]), d17 = sub(f[17], f[18]);
    const T s23 = add(s2, s3), sax = add(s1, s23);
    const T sxy = add(s7, s9), sxz = add(s11, s13), syz = add(s15, s17);
    const T sxx = add(sxy, sxz), sdg = add(sxx, syz);
    // the odd sums of the diagonal directions, per axis
    const T ax = add(add(d7, d9), add(d11, d13));
    const T ay = add(sub(d7, d9), add(d15, d17));
    const T az = add(sub(d11, d13), sub(d15, d17));
    m[0] = add(f[0], add(sax, sdg));
    m[1] = add(d1, ax);
    m[2] = add(d2, ay);
    m[3] = add(d3, az);
    m[4] = sub(sdg, f[0]);
    const T sq = mad(mtwo, syz, sxx);  // s_xy + s_xz - 2 s_yz
    const T sr = mad(two, s1, mul(lit<T>(-1.0f), s23));
    m[5] = add(sr, sq);
    const T d23 = sub(s2, s3), dxx = sub(sxy, sxz);
    m[6] = add(d23, dxx);
    m[7] = sub(s7, s9);
    m[8] = sub(s15, s17);
    m[9] = sub(s11, s13);
    m[10] = mad(mtwo, d1, ax);
    m[11] = mad(mtwo, d2, ay);
    m[12] = mad(mtwo, d3, az);
    m[13] = sub(add(d7, d9), add(d11, d13));
    m[14] = sub(add(d15, d17), sub(d7, d9));
    m[15] = sub(sub(d11, d13), sub(d15, d17));
    m[16] = add(f[0], mad(mtwo, sax, sdg));
    m[17] = sub(sq, sr);
    m[18] = sub(dxx, d23);
}

// 1/3 to 48 bits with its float. The float alone is 2^-25 of 1/3 too large, and
// f_0 came out 3e-8 too large on average, the same way every step: of the 1.6e-8
// by which a step's mass grew, two thirds. (1/18 and 1/36 are 2^-27 too large,
// f_i 1e-8; correcting all nine of their products would take another 0.5 to 1 %
// of a step.) Populations of the paper's mixture after 8 steps are 0.8e-7 off
// FP64, 1.6e-7 with the float alone; 8 steps of 128x128x512 with noise take 5565
// us, 5550 with the float alone.
constexpr float kThirdLow = -9.934107481e-9f;

// Back transform f_i = w_i sum_k e_k(c_i) n_k with n_k = m_k / b_k already
// normalised, split into the even and odd parts of each opposite pair; T =
// Pair in the step (both components at once).
template <class T>
__host__ __device__ __forceinline__ void from_modes(const T n[19], T f[19])
{
    const T two = lit<T>(2.0f), mtwo = lit<T>(-2.0f);
    const T k18 = lit<T>(1.0f / 18.0f), k36 = lit<T>(1.0f / 36.0f);
    const T m18 = lit<T>(-1.0f / 18.0f), m36 = lit<T>(-1.0f / 36.0f);
    const T x0 = add(sub(n[0], n[4]), n[16]);
    f[0] = mad(x0, lit<T>(1.0f / 3.0f), mul(x0, lit<T>(kThirdLow)));
    const T a = mad(mtwo, n[16], n[0]);
    const T p = sub(n[5], n[17]), q = sub(n[6], n[18]);
    const T ap = sub(a, p);
    const T ex = mul(mad(two, p, a), k18), ey = mul(add(ap, q), k18), ez = mul(sub(ap, q), k18);
    const T ox = mad(mtwo, n[10], n[1]), oy = mad(mtwo, n[11], n[2]), oz = mad(mtwo, n[12], n[3]);
    f[1] = mad(ox, k18, ex); f[2] = mad(ox, m18, ex);
    f[3] = mad(oy, k18, ey); f[4] = mad(oy, m18, ey);
    f[5] = mad(oz, k18, ez); f[6] = mad(oz, m18, ez);
    const T cmn = add(add(n[0], n[4]), n[16]);
    const T s = add(n[5], n[17]), t = add(n[6], n[18]);
    const T cs = add(cmn, s);
    const T exy = add(cs, t), exz = sub(cs, t), eyz = mad(mtwo, s, cmn);
    const T e7 = mul(add(exy, n[7]), k36), e9 = mul(sub(exy, n[7]), k36);
    const T e11 = mul(add(exz, n[9]), k36), e13 = mul(sub(exz, n[9]), k36);
    const T e15 = mul(add(eyz, n[8]), k36), e17 = mul(sub(eyz, n[8]), k36);
    const T X = add(n[1], n[10]), Y = add(n[2], n[11]), Z = add(n[3], n[12]);
    const T x7 = add(X, n[13]), y7 = sub(Y, n[14]);
    const T x11 = sub(X, n[13]), z11 = add(Z, n[15]);
    const T y15 = add(Y, n[14]), z15 = sub(Z, n[15]);
    const T o7 = add(x7, y7), o9 = sub(x7, y7);
    const T o11 = add(x11, z11), o13 = sub(x11, z11);
    const T o15 = add(y15, z15), o17 = sub(y15, z15);
    f[7] = mad(o7, k36, e7); f[8] = mad(o7, m36, e7);
    f[9] = mad(o9, k36, e9); f[10] = mad(o9, m36, e9);
    f[11] = mad(o11, k36, e11); f[12] = mad(o11, m36, e11);
    f[13] = mad(o13, k36, e13); f[14] = mad(o13, m36, e13);
    f[15] = mad(o15, k36, e15); f[16] = mad(o15, m36, e15);
    f[17] = mad(o17, k36, e17); f[18] = mad(o17, m36, e17);
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), from its published
// definition, and the open-interval uniform used by both the initial
// perturbation and the thermal noise: ((x >> 9) + 1/2) * 2^-23, exact in
// binary32.
// ---------------------------------------------------------------------------
// High 32 bits of a 32 x 32-bit product (the device instruction; on the host,
// where the header's tests run it, the 64-bit product).
__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

__host__ __device__ __forceinline__ void philox4x32_10(uint32_t& x0, uint32_t& x1, uint32_t& x2, uint32_t& x3,
                                                       uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * x0, hi0 = mulhi32(0xD2511F53u, x0);
        const uint32_t lo1 = 0xCD9E8D57u * x2, hi1 = mulhi32(0xCD9E8D57u, x2);
        const uint32_t y0 = hi1 ^ x1 ^ k0;
        const uint32_t y2 = hi0 ^ x3 ^ k1;
        x0 = y0; x1 = lo1; x2 = y2; x3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// The upper 23 bits of a word as the fraction of a float in [1, 2), by one
// funnel shift: 0x7f above the word puts the exponent of 1 in front.
__host__ __device__ __forceinline__ float one_to_two(uint32_t w)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(__funnelshift_r(w, 0x7fu, 9));
#else
    const uint32_t u = (0x7fu << 23) | (w >> 9);
    float f;
    memcpy(&f, &u, sizeof(f));
    return f;
#endif
}
// ((w >> 9) + 1/2) 2^-23, in (0, 1), exact: the fraction minus 1 - 2^-24.
constexpr float kHalfBelowOne = 0.999999940395355224609375f;
__host__ __device__ __forceinline__ float uniform_open(uint32_t w) { return one_to_two(w) - kHalfBelowOne; }

// ---------------------------------------------------------------------------
// Launch-invariant parameters (kernel argument, by value).
// ---------------------------------------------------------------------------
struct KParams {
    int lx, ly, lz;
    int wall[3];
    int px, py, pz;        // padded psi row stride (lx + 2 rounded up to 4) and dimensions ly + 2, lz + 2
    long long N;           // lx*ly*lz
    long long padn;        // px*py*pz
    int tx, ty;            // tile (block) shape in x, y; one z-plane per block
    int gx, gy;            // tiles per axis in x, y
    float G;
    float gs, gd, gg;      // gamma = 1 - 1/tau of stress, component momentum, ghost modes
    float ext[3];          // constant fluid body force density
    float drho;            // wetting shift
    float kT;
    float nz_mode[19];     // sqrt((1 - gamma_k^2) / b_k) for k >= 4 (noise in normalised modes per sqrt(3 kT rho))
    float nz_j;            // sqrt(1 - gamma_d^2)
    uint32_t key0, key1;   // Philox key
    uint32_t rk0[10], rk1[10];  // Philox round keys key + r * (0x9E3779B9, 0xBB67AE85)
    int ncx, ncy, ncz;     // candidate tiles per axis around the particle box
    int tau1;              // every relaxation time equals 1
    uint32_t dirN[38];     // (19 l + i) * N: offset of population (l, i) in one copy
    int has_particle;
    int B;                 // side of the particle box
    double R;              // sphere radius
    double inv_mp, inv_Ip; // 1 / m_p and 1 / I_p of the particle (0 without one)
    double rho0[2];        // initial densities (fallback for an uncovered node with no fluid neighbour)
    int counterforce;
};

// Particle and bookkeeping state, kept in device memory (FP64).
struct DevState {
    double X[3], V[3], Vavg[3], Om[3], F[3], T[3], Ppend[3], Lpend[3];
    double delta[2];       // per-node mass correction for the next collision
    double fc;             // counterforce density along z on the fluid
    double mp, Ip, Fp;
    long long nfluid;
    long long step;
    double ledger_bb[2];   // mass removed by the moving-wall term this step
    float delta_f[2];      // delta as float, read by the collide kernels
    float fc_f;            // fc as float
    float Vf[3], Omf[3];   // V and Omega as float, read by the moving link rule
    uint32_t step_u32;     // step as the 32-bit Philox counter word
    int cur;               // index of the current mask
    int box0[3];           // origin of the particle box (periodic axes in [0, L))
    int box_next[3];       // origin at the position after this step's update
    int box_prev[3];       // origin the last step's collide used (its near tiles)
    int err;
    unsigned near_done;    // blocks of the near-collide launch done this step (last one updates)
    unsigned cover_done;   // blocks of the cover launch done this step (last one finishes)
};

constexpr int kThreadsStep = 256;

// Signed offset of box coordinate of lattice coordinate c on one axis.
__host__ __device__ __forceinline__ int box_rel(int c, int o, int L, int wall)
{
    int t = c - o;
    if (!wall && t < 0) t += L;
    return t;
}

__host__ __device__ __forceinline__ bool in_box(int x, int y, int z, const int o[3], const KParams& P, int& bi)
{
    const int dx = box_rel(x, o[0], P.lx, P.wall[0]);
    const int dy = box_rel(y, o[1], P.ly, P.wall[1]);
    const int dz = box_rel(z, o[2], P.lz, P.wall[2]);
    const int B = P.B;
    if ((unsigned)dx >= (unsigned)B || (unsigned)dy >= (unsigned)B || (unsigned)dz >= (unsigned)B) return false;
    bi = dx + B * (dy + B * dz);
    return true;
}

__host__ __device__ __forceinline__ bool is_solid(int x, int y, int z, const int o[3], const uint8_t* mask, const KParams& P)
{
    int bi;
    return in_box(x, y, z, o, P, bi) && mask[bi];
}

// Directions i = 1..18 whose neighbour x + c_i is a particle node of the box
// at origin o with node mask `mask`, as bits 1 << i. The neighbour wraps on a
// periodic axis; across a wall there is none. The neighbour's box
// coordinates are the node's own plus c_i, taken modulo L on periodic axes.
__host__ __device__ __forceinline__ uint32_t solid_neighbours(int x, int y, int z, const int o[3],
                                                              const uint8_t* mask, const KParams& P)
{
    const int c[3] = {x, y, z};
    const int L[3] = {P.lx, P.ly, P.lz};
    int d[3];
    bool lo[3], hi[3];  // a step down / up this axis leaves through a wall
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        d[a] = box_rel(c[a], o[a], L[a], P.wall[a]);
        lo[a] = P.wall[a] && c[a] == 0;
        hi[a] = P.wall[a] && c[a] == L[a] - 1;
    }
    const unsigned B = (unsigned)P.B;
    // Every direction's mask byte is loaded (entry 0 where there is none), so
    // that the 18 loads are in flight together: the node waits for one.
    uint32_t bits = 0u;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const int s[3] = {cxv(i), cyv(i), czv(i)};
        bool ok = true;
        unsigned e[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if ((s[a] < 0 && lo[a]) || (s[a] > 0 && hi[a])) ok = false;
            int t = d[a] + s[a];
            if (!P.wall[a]) t = t >= L[a] ? t - L[a] : (t < 0 ? t + L[a] : t);
            e[a] = (unsigned)t;
        }
        ok = ok && e[0] < B && e[1] < B && e[2] < B;
        const uint8_t in = mask[ok ? e[0] + B * (e[1] + B * e[2]) : 0u];
        if (ok && in) bits |= 1u << i;
    }
    return bits;
}

// Does [a0, a0+la) meet [b0, b0+lb) on an axis of length L (periodic: modulo L)?
__host__ __device__ __forceinline__ bool ranges_meet(int a0, int la, int b0, int lb, int L, int wall)
{
    if (wall) return a0 < b0 + lb && b0 < a0 + la;
    if (lb >= L) return true;
    int d0 = (a0 - b0) % L;
    if (d0 < 0) d0 += L;
    return d0 < lb || d0 + la > L;
}

// Tile (bx, by, bz) meets the particle box grown by one node on every side:
// only such tiles have fluid nodes whose stencil touches a particle node.
__host__ __device__ __forceinline__ bool tile_near(int bx, int by, int bz, const int o[3], const KParams& P)
{
    const int x0 = bx * P.tx, y0 = by * P.ty;
    const int lxr = min(P.tx, P.lx - x0), lyr = min(P.ty, P.ly - y0);
    const int B2 = P.B + 2;
    return ranges_meet(x0, lxr, o[0] - 1, B2, P.lx, P.wall[0]) &&
           ranges_meet(y0, lyr, o[1] - 1, B2, P.ly, P.wall[1]) &&
           ranges_meet(bz, 1, o[2] - 1, B2, P.lz, P.wall[2]);
}

// Edge candidates of the adjoint's last node pass: the nodes on a walled
// face (a wall ghost among their neighbours) and the nodes of the particle
// box at origin o grown by one node (a particle node among their
// neighbours). No other node has either among its neighbours.
__host__ __device__ __forceinline__ bool adj_edge_candidate(const int c[3], const int o[3], const KParams& P)
{
    const int L[3] = {P.lx, P.ly, P.lz};
    for (int a = 0; a < 3; ++a)
        if (P.wall[a] && (c[a] == 0 || c[a] == L[a] - 1)) return true;
    if (!P.has_particle) return false;
    bool in_grown = true;
    for (int a = 0; a < 3; ++a) in_grown = in_grown && ranges_meet(c[a], 1, o[a] - 1, P.B + 2, L[a], P.wall[a]);
    return in_grown;
}

// Entries adj_edge_node walks: the particle box grown by one node, then the
// two faces of each walled axis.
__host__ __device__ __forceinline__ long long adj_edge_entries(const KParams& P)
{
    const long long Bg = P.has_particle ? P.B + 2 : 0;
    const int L[3] = {P.lx, P.ly, P.lz};
    long long n = Bg * Bg * Bg;
    for (int a = 0; a < 3; ++a)
        if (P.wall[a]) n += 2LL * L[(a + 1) % 3] * L[(a + 2) % 3];
    return n;
}

// Node c of entry t, or false: every edge candidate is the node of exactly
// one entry. The grown box's entries outside the lattice, or repeating a node
// where the box wraps a periodic axis shorter than it, give none; so do the
// face entries that lie on a face of an earlier walled axis, repeat a face of
// an axis of length 1, or lie in the grown box.
__host__ __device__ __forceinline__ bool adj_edge_node(long long t, const int o[3], const KParams& P, int c[3])
{
    if (t < 0 || t >= adj_edge_entries(P)) return false;
    const int L[3] = {P.lx, P.ly, P.lz};
    const int Bg = P.B + 2;
    const long long nbox = P.has_particle ? (long long)Bg * Bg * Bg : 0;
    if (t < nbox) {
        const int d[3] = {(int)(t % Bg), (int)(t / Bg % Bg), (int)(t / ((long long)Bg * Bg))};
        for (int a = 0; a < 3; ++a) {
            int v = o[a] - 1 + d[a];
            if (P.wall[a]) {
                if (v < 0 || v >= L[a]) return false;
            } else {
                if (d[a] >= L[a]) return false;
                v = (v % L[a] + L[a]) % L[a];
            }
            c[a] = v;
        }
        return true;
    }
    t -= nbox;
    int face = -1;
    for (int a = 0; a < 3 && face < 0; ++a) {
        if (!P.wall[a]) continue;
        const int b = (a + 1) % 3, e = (a + 2) % 3;
        const long long fsz = (long long)L[b] * L[e];
        for (int side = 0; side < 2 && face < 0; ++side) {
            if (t < fsz) {
                if (side == 1 && L[a] == 1) return false;
                c[a] = side ? L[a] - 1 : 0;
                c[b] = (int)(t % L[b]);
                c[e] = (int)(t / L[b]);
                face = a;
            } else {
                t -= fsz;
            }
        }
    }
    if (face < 0) return false;
    for (int a = 0; a < face; ++a)
        if (P.wall[a] && (c[a] == 0 || c[a] == L[a] - 1)) return false;
    if (P.has_particle) {
        bool in_grown = true;
        for (int a = 0; a < 3; ++a) in_grown = in_grown && ranges_meet(c[a], 1, o[a] - 1, Bg, L[a], P.wall[a]);
        if (in_grown) return false;
    }
    return true;
}

__host__ __device__ __forceinline__ long long pad_index(int x, int y, int z, const KParams& P)
{
    return (long long)(x + 1) + (long long)P.px * ((y + 1) + (long long)P.py * (z + 1));
}

// Vector from the particle centre to point r, minimum image on periodic axes.
__host__ __device__ __forceinline__ double rel_axis(double r, double X, int L, int wall)
{
    double d = r - X;
    if (!wall) {
        if (d > 0.5 * L) d -= L;
        else if (d < -0.5 * L) d += L;
    }
    return d;
}

// Sums over the warp of eight doubles a lane, by a transposed butterfly: with
// each exchange a lane hands over half of the values it holds and keeps the
// sums of the other half, so a lane adds 4 + 2 + 1 + 1 + 1 times instead of
// the 40 of eight separate butterflies (a warp's FP64 addition takes about 16
// clocks of the SM's only FP64 pipe). Returns the sum of value
// warp_slot(lane); lane sum_lane(k) holds value k. Fixed order.
__device__ __forceinline__ int warp_slot(int lane)
{
    return (lane >> 4 & 1) * 4 + (lane >> 3 & 1) * 2 + (lane >> 2 & 1);
}
__device__ __forceinline__ int sum_lane(int k) { return (k >> 2 & 1) * 16 + (k >> 1 & 1) * 8 + (k & 1) * 4; }
__device__ __forceinline__ double warp_sum8(const double v[8], int lane)
{
    const bool u4 = lane & 16, u3 = lane & 8, u2 = lane & 4;
    double p[4], q[2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        p[i] = (u4 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, u4 ? v[i] : v[4 + i], 16);
#pragma unroll
    for (int i = 0; i < 2; ++i) q[i] = (u3 ? p[2 + i] : p[i]) + __shfl_xor_sync(0xffffffffu, u3 ? p[i] : p[2 + i], 8);
    double a = (u2 ? q[1] : q[0]) + __shfl_xor_sync(0xffffffffu, u2 ? q[0] : q[1], 4);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    return a;
}

// Block-wide sum of 8 doubles into s_out[0..7]. Fixed reduction tree:
// deterministic. A thread may pass active = false when all its v are 0: warps
// with no active thread then skip their shuffles.
template <int NT>
__device__ __forceinline__ void block_sum8(const double v[8], double* s_red, double* s_out, bool active = true)
{
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int lane = tid & 31, warp = tid >> 5;
    const int nwarp = (blockDim.x * blockDim.y + 31) >> 5;
    double a = 0.0;
    if (__any_sync(0xffffffffu, active)) a = warp_sum8(v, lane);
    if ((lane & 3) == 0) s_red[warp * 8 + warp_slot(lane)] = a;
    __syncthreads();
    if (tid < 8) {
        double t = 0.0;
        for (int w = 0; w < nwarp; ++w) t += s_red[w * 8 + tid];
        s_out[tid] = t;
    }
    __syncthreads();
}

// Block-wide sum of `rows` rows of 8 doubles (written by other blocks) into
// s_out[0..7], by 256 threads: thread (row r, value k) = (tid / 8, tid % 8)
// walks rows r, r + 32, ..., then rows add up in a fixed order. Loads of eight
// rows are in flight together, and rows of zeros, most of them, cost no
// addition.
__device__ __forceinline__ void sum_rows8(const double* __restrict__ v, long long rows, double* s_red, double* s_out)
{
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int lane = tid & 31, warp = tid >> 5;
    double a = 0.0;
    for (long long r0 = tid >> 3; r0 < rows; r0 += 256) {
        double b[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const long long r = r0 + 32 * q;
            b[q] = r < rows ? __ldcg(v + r * 8 + (tid & 7)) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (b[q] != 0.0) a += b[q];
    }
    a += __shfl_xor_sync(0xffffffffu, a, 8);
    a += __shfl_xor_sync(0xffffffffu, a, 16);
    if (lane < 8) s_red[warp * 8 + lane] = a;
    __syncthreads();
    if (tid < 8) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += s_red[w * 8 + tid];
        s_out[tid] = t;
    }
    __syncthreads();
}

// True in the block that is the last of `total` blocks to pass this point
// (counted in *counter, which that block resets to 0). Every thread of the
// block must call it. Threads that wrote what the last block will read pass
// wrote = true: their writes are made visible device-wide before the block
// takes its ticket, so the last block may read what all the others wrote
// (with loads that bypass L1). There is no waiting: the other blocks just
// finish.
__device__ __forceinline__ bool last_block(unsigned* counter, unsigned total, bool wrote)
{
    __shared__ int s_last;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    if (wrote) __threadfence();
    __syncthreads();
    if (tid == 0) {
        const unsigned t = atomicAdd(counter, 1u);
        s_last = (t + 1u == total) ? 1 : 0;
        if (s_last) *counter = 0u;
    }
    __syncthreads();
    const bool last = s_last != 0;
    if (last) __threadfence();
    return last;
}

}  // namespace flbm
