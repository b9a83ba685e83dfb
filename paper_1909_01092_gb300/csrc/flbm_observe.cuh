// Observables of a state (declared in include/flbm.h as flbm_observables):
// masses, momentum and kinetic energy over the fluid nodes, and the sums
// behind the mode, interdiffusion and momentum temperatures over the bulk
// fluid nodes (arXiv:1909.01092, Section 2, fluctuation-dissipation), in FP64.
//
// One pass reads every population once. A block of 128 threads walks a column
// of nodes over K planes, keeps its 48 sums in registers and adds them up once
// at the end; a second launch adds the blocks' sums. The FP64 pipe (a warp's
// instruction holds it for about 16 clocks) bounds the pass, by some 300
// operations a node: a call on 128x128x128 takes 1.23 ms, against 3.62 ms in
// two passes with every sum reduced per tile. Double-floats would take 0.34 ms,
// but their 48 bits show in the result: against 113 bits, the temperatures of
// thermal states are 1.5e-15 off (FP64: 4e-16) and diff_temp of a noise-free
// flow, whose components move together, 2e-13 (FP64: 4e-16); and they need a
// bound on the velocity as well as on the populations.
#pragma once

#include <algorithm>

#include "flbm_kernels.cuh"

namespace flbm {

// A block's sums:
//   2 (k - 4) + l for k = 4..18 and l = A, B: n_lk^2 (bulk), n_lk = m_lk - m_lk^eq(rho_l, u), u = j / rho_tot
//   30 + l: rho_l (bulk)   32 + l: rho_l (fluid)
//   34 + 2 a, 35 + 2 a: d_a^2, j_a^2 (bulk), d = (rho_B j_A - rho_A j_B) / rho_tot, j = j_A + j_B
//   40: rho_A rho_B / rho_tot (bulk)   41: j^2 / (2 rho_tot) (fluid)
//   42 + a: j_a (fluid)   45: bulk nodes   46: non-finite populations   47: unused
constexpr int kObsValues = 48;
constexpr int kObsThreads = 128;
constexpr int kObsBlocks = 2;  // resident per SM: a thread's sums alone take 96 registers

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
    // As many planes as leave eight blocks for each resident one, up to 16: a
    // block's 48 sums cost as much as a sixth of a plane.
    const long long planes = (long long)P.gx * g.gy * P.lz;
    g.K = (int)std::clamp(planes / (8LL * kObsBlocks * 152), 1LL, 16LL);
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

static __global__ void __launch_bounds__(kObsThreads, kObsBlocks)
    k_obs(const float* __restrict__ f, const DevState* __restrict__ st, const uint8_t* __restrict__ masks,
          double* __restrict__ parts, KParams P, ObsGeom G)
{
    const long long block = blockIdx.x + (long long)gridDim.x * blockIdx.y;
    const int by = blockIdx.x / P.gx, bx = blockIdx.x - by * P.gx;
    const int tx = threadIdx.x & (P.tx - 1), ty = threadIdx.x >> (__ffs(P.tx) - 1);
    const int x = bx * P.tx + tx, y = by * G.rows + ty;
    const int z0 = blockIdx.y * G.K, z1 = min(z0 + G.K, P.lz);
    double acc[kObsValues];
#pragma unroll
    for (int k = 0; k < kObsValues; ++k) acc[k] = 0.0;
    int bad = 0;  // non-finite populations
    if (x < P.lx && y < P.ly) {
        for (int z = z0; z < z1; ++z) {
            bool fluid, bulk;
            observe_kind(x, y, z, st, masks, P, fluid, bulk);
            if (!fluid) continue;
            const uint32_t n = (uint32_t)x + (uint32_t)P.lx * ((uint32_t)y + (uint32_t)P.ly * (uint32_t)z);
            float v[38];
#pragma unroll
            for (int q = 0; q < 38; ++q) v[q] = __ldg(at(f + P.dirN[q], 4u * n));
            double m[2][19];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                double fl[19];
#pragma unroll
                for (int i = 0; i < 19; ++i) {
                    bad += !isfinite(v[19 * l + i]);
                    fl[i] = (double)v[19 * l + i];
                }
                to_modes(fl, m[l]);
                acc[32 + l] += m[l][0];
            }
            const double rt = m[0][0] + m[1][0];
            const double j[3] = {m[0][1] + m[1][1], m[0][2] + m[1][2], m[0][3] + m[1][3]};
            const double u[3] = {j[0] / rt, j[1] / rt, j[2] / rt};
            acc[42] += j[0];
            acc[43] += j[1];
            acc[44] += j[2];
            acc[41] += rt > 0.0 ? 0.5 * (j[0] * u[0] + j[1] * u[1] + j[2] * u[2]) : 0.0;
            if (!bulk) continue;
            const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
            const double eq[6] = {uu, 3.0 * u[0] * u[0] - uu, u[1] * u[1] - u[2] * u[2],
                                  u[0] * u[1], u[1] * u[2], u[0] * u[2]};
#pragma unroll
            for (int l = 0; l < 2; ++l) {
#pragma unroll
                for (int k = 4; k < 19; ++k) {
                    const double nk = k <= 9 ? m[l][k] - m[l][0] * eq[k - 4] : m[l][k];
                    acc[2 * (k - 4) + l] += nk * nk;
                }
                acc[30 + l] += m[l][0];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double d = (m[1][0] * m[0][1 + a] - m[0][0] * m[1][1 + a]) / rt;
                acc[34 + 2 * a] += d * d;
                acc[35 + 2 * a] += j[a] * j[a];
            }
            acc[40] += m[0][0] * m[1][0] / rt;
            acc[45] += 1.0;
        }
    }
    acc[46] = (double)bad;
    __shared__ double s_red[(kObsThreads / 32) * 8];
    __shared__ double s_out[8];
#pragma unroll
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
inline cudaError_t launch_observe(const float* f, const DevState* st, const uint8_t* masks, double* parts, ObsOut* out,
                                  const KParams& P, cudaStream_t s)
{
    const ObsGeom G = obs_geom(P);
    const dim3 grid(P.gx * G.gy, G.nz);
    k_obs<<<grid, kObsThreads, 0, s>>>(f, st, masks, parts, P, G);
    k_obs_sum<<<kObsValues, 256, 0, s>>>(parts, G.blocks, st, out);
    return cudaGetLastError();
}

}  // namespace flbm
