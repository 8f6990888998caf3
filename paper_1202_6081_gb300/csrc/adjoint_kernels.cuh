// Kernels of the discrete adjoint of the step (D3Q27 and D3Q15) and of the
// seeds of the objectives (not in the paper: the reverse mode of its update).
//
// Forward step (pull form): f_{t+1}[a](x) = C_a(f_t(x - e_a)), or, behind a
// bounce-back wall, C_opp(a)(f_t(x)).  Its transpose for the adjoint
// lam = dJ/df:
//     lam_t(y) = J_C(f_t(y))^T mu(y),   mu_b(y) = lam_{t+1}[b](y + e_b)
// (or lam_{t+1}[opp b](y) when y + e_b is behind a wall), and
//     dJ/dF(y) += (dC/dF)^T mu(y).
// Adjoint fields are FP32, laid out like the state (population planes of
// pitched rows).
#pragma once

#include "adjoint_q15.cuh"
#include "adjoint_q27.cuh"
#include "kernels.cuh"

namespace lbm {

// Per-cell reverse of the collision, chosen by the lattice (array size).
// kEq: the rate-1 form (D3Q27).
template <bool kEq, typename V>
__device__ __forceinline__ void adjoint_collide(const V (&f)[27], V Fx, V Fy, V Fz,
                                                const Rates27<V> &r, const V (&mu)[27],
                                                V (&lam)[27], V &gx, V &gy, V &gz) {
    adjoint27<kEq, V>(f, Fx, Fy, Fz, r, mu, lam, gx, gy, gz);
}
template <bool, typename V>
__device__ __forceinline__ void adjoint_collide(const V (&f)[15], V Fx, V Fy, V Fz,
                                                const Rates15<V> &r, const V (&mu)[15],
                                                V (&lam)[15], V &gx, V &gy, V &gz) {
    adjoint15<V>(f, Fx, Fy, Fz, r, mu, lam, gx, gy, gz);
}

// The rates of lattice Q in both lanes, from the host-built PackedRates.
template <int Q>
struct PairRates;
template <>
struct PairRates<27> {
    using type = Rates27<f2>;
    static __device__ __forceinline__ type load(const PackedRates &p) {
        return load_rates_packed(p);
    }
};
template <>
struct PairRates<15> {
    using type = Rates15<f2>;
    static __device__ __forceinline__ type load(const PackedRates &p) {
        Rates15<f2> r;
#pragma unroll
        for (int b = 0; b < 15; ++b) r.w[b] = f2(p.w15[b]);
        return r;
    }
};

struct AdjointArgs {
    const float *lam_next[27];  // planes of lam_{t+1} (the first Q used)
    float *lam_out[27];         // planes of lam_t
    float *gF;                  // dense [3][N] accumulator or nullptr
};

// The adjoint step, one cell per thread, for small grids with rows of odd length
// (see step1_kernel); the adjoint is pulled from the mirrored neighbours x + e_q.
template <int Q, typename T, bool kWalls, bool kEq>
__global__ void __launch_bounds__(128) adjoint1_kernel(const StepIO<T> io, const AdjointArgs g,
                                                       const StepArgs a) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    const int xs[3] = {(x + 1 == a.g.nx) ? 0 : x + 1, x, (x == 0) ? a.g.nx - 1 : x - 1};
    float f[Q], mu[Q];
    pull_cell<Q, T, false>(io, R, x, a.g.nx, f);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr int i = ex<Q>(q) + 1, j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
        const bool wall = kWalls && R.wall[2 - j][2 - k];
        const int src = wall ? R.own + x : R.off[2 - j][2 - k] + xs[2 - i];
        mu[q] = Pair<float>::ld1(element<false>(g.lam_next[wall ? opposite<Q>(q) : q], src));
    });
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, x, y, z);
    float Fx, Fy, Fz;
    cell_force(a, c, N, Fx, Fy, Fz);
    const typename Rates<Q>::type r = load_rates<Q>(a);
    float lam[Q], gF[3];
    adjoint_collide<kEq, float>(f, Fx, Fy, Fz, r, mu, lam, gF[0], gF[1], gF[2]);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        __stcs(element<false>(g.lam_out[q], R.own + x), lam[q]);
    });
    if (g.gF) {
#pragma unroll
        for (int d = 0; d < 3; ++d) g.gF[d * N + c] += gF[d];
    }
}

// The pair's adjoints of its post-collision values, from the mirrored
// neighbours; kSel: with the wall selects.
template <int Q, bool kSel, bool kWalls, bool kRag>
__device__ __forceinline__ void pull_adjoint(const AdjointArgs &g, const Rows<kWalls> &R,
                                             const PairCols<kRag> &X, f2 (&mu)[Q]) {
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr int i = ex<Q>(q), j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
        if (kSel && R.wall[2 - j][2 - k]) {
            mu[q] = Pair<float>::ld2(element<kRag>(g.lam_next[opposite<Q>(q)], R.own + X.x0));
        } else {
            mu[q] = ld_shifted(g.lam_next[q], R.off[2 - j][2 - k], -i, X);
        }
    });
}

// The adjoint step for two neighbouring cells (x0, x0 + 1) per thread in
// packed f32x2 arithmetic.  The state is pulled as in step2_kernel; the adjoint
// is pulled from the mirrored neighbours x + e_q: for e_x = 0 an aligned pair,
// for e_x = +1 the cells (x0 + 1, x0 + 2), for e_x = -1 (x0 - 1, x0).
// Bound by HBM: 360 bytes per cell (D3Q27 FP32 with a force field and dJ/dF).
// 3 blocks of 128 threads per SM, 168 registers: D3Q15 fits without spills;
// D3Q27 at general rates spills ~100 B (121 us at 128^3; 4 blocks spill ~700 B,
// 206 us).  The rate-1 form (kEq, adjoint27) needs fewer and takes 4 blocks, 128
// registers: 128^3 in 113.8 us, 6.64 TB/s, where the general form took 135; FP16
// states 114 / 119 us at 4 / 3 blocks; 3 blocks for BF16 states (117 / 126 at 4)
// and ragged rows (126 x 128 x 128 walled 122 / 127).
// kRag: ragged rows (PairCols).
template <typename T, bool kRag, bool kEq>
constexpr int kAdjointBlocks = kEq && !kRag && !Storage<T>::kRef ? 4 : 3;

template <int Q, typename T, bool kWalls, bool kRag, bool kEq>
__global__ void __launch_bounds__(128, (kAdjointBlocks<T, kRag, kEq>)) adjoint2_kernel(const StepIO<T> io, const AdjointArgs g,
                                                       const StepArgs a, const PackedRates pr) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (2 * t >= row_end<float, kRag>(a.g.nx) || y >= a.g.ny) return;
    const PairCols<kRag> X(2 * t, a.g.nx);
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    f2 f[Q], mu[Q];
    pull_pairs<Q, T>(io, R, X, f);
    if (kWalls && (R.edge || blockDim.x < 32))
        pull_adjoint<Q, kWalls>(g, R, X, mu);
    else
        pull_adjoint<Q, false>(g, R, X, mu);
    // deviations f - w: 16-bit values scaled by w
    if constexpr (Storage<T>::kScaled) {
        static_for<Q>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            f[q] = f[q] * f2(float(weight<Q>(q)));
        });
    }
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, X.x0, y, z);
    f2 Fx, Fy, Fz;
    pair_force(a, X, y, z, Fx, Fy, Fz);
    // the dJ/dF accumulator is read now, so its latency hides behind the
    // collision's reverse; it is written back at the end.  A thread that repeats
    // the last pair leaves it to that pair's own thread, which overwrites it.
    f2 acc[3] = {f2(0.0f), f2(0.0f), f2(0.0f)};
    if (g.gF && X.owner()) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float *p = g.gF + d * N + c;
            acc[d] = f2(p[0], p[X.single() ? 0 : 1]);
        }
    }
    const typename PairRates<Q>::type r = PairRates<Q>::load(pr);
    f2 lam[Q], gF[3];
    adjoint_collide<kEq, f2>(f, Fx, Fy, Fz, r, mu, lam, gF[0], gF[1], gF[2]);
    zero_padding(X, lam);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        Pair<float>::st2(element<kRag>(g.lam_out[q], R.own + X.at), lam[q]);
    });
    if (g.gF && X.owner()) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float *p = g.gF + d * N + c;
            acc[d] = acc[d] + gF[d];
            p[0] = acc[d].lo();
            if (!X.single()) p[1] = acc[d].hi();
        }
    }
}

// Seed of the adjoint for J = sum_x rho |u|^2 / 2 at the final state:
// lam_a = u.e_a - |u|^2 / 2, and the direct term dJ/dF += u / 2
// (u = (j + F/2) / rho).
template <int Q, typename T>
__global__ void __launch_bounds__(128) energy_seed_kernel(const StepIO<T> io,
                                                          const StepArgs a, AdjointArgs g) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    float f[Q];
    gather<Q, T>(io, a.g, x, y, z, f);
    float drho, jx, jy, jz, Fx, Fy, Fz;
    moments<Q>(f, drho, jx, jy, jz);
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, x, y, z);
    cell_force(a, c, N, Fx, Fy, Fz);
    const float ir = 1.0f / (1.0f + drho);
    const float ux = (jx + 0.5f * Fx) * ir, uy = (jy + 0.5f * Fy) * ir, uz = (jz + 0.5f * Fz) * ir;
    const float h = 0.5f * (ux * ux + uy * uy + uz * uz);
    const long long own = ((long long)z * a.g.ny + y) * a.g.px + x;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        g.lam_out[q][own] = ex<Q>(q) * ux + ey<Q>(q) * uy + ez<Q>(q) * uz - h;
    if (g.gF) {
        g.gF[c] += 0.5f * ux;
        g.gF[N + c] += 0.5f * uy;
        g.gF[2 * N + c] += 0.5f * uz;
    }
}

// Seed of the adjoint for an objective J(rho, u) of the macroscopic fields
// (Eqs. densitycalculation, velocitycalculation) given g_rho = dJ/drho and
// g_u = dJ/du per cell (dense FP32; NULL = zero): since d rho / d f_a = 1 and
// d u_i / d f_a = (e_ai - u_i) / rho,
//     lam_a = g_rho + sum_i (e_ai - u_i) g_u_i / rho,
// and the direct term dJ/dF_i += g_u_i / (2 rho) (u carries F/2).
template <int Q, typename T>
__global__ void __launch_bounds__(128) macro_seed_kernel(const StepIO<T> io,
                                                         const StepArgs a, AdjointArgs g,
                                                         const float *__restrict__ g_rho,
                                                         const float *__restrict__ g_u) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    float f[Q];
    gather<Q, T>(io, a.g, x, y, z, f);
    float drho, jx, jy, jz, Fx, Fy, Fz;
    moments<Q>(f, drho, jx, jy, jz);
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, x, y, z);
    cell_force(a, c, N, Fx, Fy, Fz);
    const float ir = 1.0f / (1.0f + drho);
    const float ux = (jx + 0.5f * Fx) * ir, uy = (jy + 0.5f * Fy) * ir, uz = (jz + 0.5f * Fz) * ir;
    const float gr = g_rho ? g_rho[c] : 0.0f;
    const float gx = g_u ? g_u[c] * ir : 0.0f;
    const float gy = g_u ? g_u[N + c] * ir : 0.0f;
    const float gz = g_u ? g_u[2 * N + c] * ir : 0.0f;
    const float base = gr - (ux * gx + uy * gy + uz * gz);
    const long long own = ((long long)z * a.g.ny + y) * a.g.px + x;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        g.lam_out[q][own] = base + ex<Q>(q) * gx + ey<Q>(q) * gy + ez<Q>(q) * gz;
    if (g.gF) {
        g.gF[c] += 0.5f * gx;
        g.gF[N + c] += 0.5f * gy;
        g.gF[2 * N + c] += 0.5f * gz;
    }
}

// Per-block partial sums of rho |u|^2 / 2 (slot 0 of each 4-double record),
// cells assigned to blocks as in the conservation reduction.
template <int Q, typename T>
__global__ void __launch_bounds__(128, 8) energy_kernel(const StepIO<T> io, const StepArgs a,
                                                        double *__restrict__ part) {
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    double acc[1] = {0.0};
    for_cells(a.g, [&](int x, int y, int z, long long c) {
        float f[Q];
        gather<Q, T>(io, a.g, x, y, z, f);
        float drho, jx, jy, jz, Fx, Fy, Fz;
        moments<Q>(f, drho, jx, jy, jz);
        cell_force(a, c, N, Fx, Fy, Fz);
        const float px = jx + 0.5f * Fx, py = jy + 0.5f * Fy, pz = jz + 0.5f * Fz;
        acc[0] += widen(0.5f * (px * px + py * py + pz * pz) / (1.0f + drho));
    });
    block_sum(acc);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        part[4 * blockIdx.x] = acc[0];
        part[4 * blockIdx.x + 1] = 0.0;
        part[4 * blockIdx.x + 2] = 0.0;
        part[4 * blockIdx.x + 3] = 0.0;
    }
}

// Grids of odd rows take the one-cell adjoint kernel up to this many warps on an SM
// (kOneCellWarps).  us a step, one / two cells per thread, FP32, periodic / walled:
// D3Q27 at general rates 21^3 (4 warps) 4.17 / 6.09, 29^3 (8) 5.18 / 6.61, 33^3 (16)
// 6.59 / 6.47; walled 4.49 / 6.06, 5.34 / 6.44, 7.47 / 6.91; D3Q15 periodic 21^3 3.50 /
// 3.91, 29^3 4.00 / 4.14, walled 3.65 / 3.86, 4.15 / 4.00.
template <int Q>
constexpr int kOneCellAdjointWarps = Q == 27 ? 8 : 4;

template <int Q, typename T>
cudaError_t launch_adjoint(const void *f_t, const float *lam_next, float *lam_out, float *gF,
                           const StepArgs &a, cudaStream_t st) {
    const StepIO<T> io = step_io<Q, T>(f_t, nullptr, a.g);
    AdjointArgs g{};
    for (int q = 0; q < Q; ++q) {
        g.lam_next[q] = lam_next + q * a.g.pop;
        g.lam_out[q] = lam_out + q * a.g.pop;
    }
    g.gF = gF;
    const CellLaunch one = cell_launch(a.g);
    const bool one_cell =
        a.g.nx % 2 && a.g.nx > 1 && one.sm_warps() <= kOneCellAdjointWarps<Q>;
    const CellLaunch L = pair_launch(a.g, stored_row<float>(a.g.nx));
    const PackedRates pr = packed_rates(a);
    // ragged periodic rows without the wall selects (us a step, FP32, with / without:
    // D3Q27 30^3 5.8 / 3.8, at general rates 6.5 / 4.8, 126 x 128 x 128 120 / 117; D3Q15
    // 30^3 4.0 / 3.4), but not D3Q15 in longer rows (126 x 128 x 128 82.6 / 100)
    const bool periodic_form = Q == 27 || L.block.x < 32;
    const auto launch = [&](auto eq) {
        constexpr bool kEq = decltype(eq)::value;
        if (one_cell && a.g.bc)
            adjoint1_kernel<Q, T, true, kEq><<<one.grid, one.block, 0, st>>>(io, g, a);
        else if (one_cell)
            adjoint1_kernel<Q, T, false, kEq><<<one.grid, one.block, 0, st>>>(io, g, a);
        else if (ragged<float>(a.g) && (a.g.bc || !periodic_form))
            adjoint2_kernel<Q, T, true, true, kEq><<<L.grid, L.block, 0, st>>>(io, g, a, pr);
        else if (ragged<float>(a.g))
            adjoint2_kernel<Q, T, false, true, kEq><<<L.grid, L.block, 0, st>>>(io, g, a, pr);
        else if (a.g.bc)
            adjoint2_kernel<Q, T, true, false, kEq><<<L.grid, L.block, 0, st>>>(io, g, a, pr);
        else
            adjoint2_kernel<Q, T, false, false, kEq><<<L.grid, L.block, 0, st>>>(io, g, a, pr);
    };
    if constexpr (Q == 27) {
        if (higher_rates_are_one(a)) {
            launch(std::true_type{});
            return cudaGetLastError();
        }
    }
    launch(std::false_type{});
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_energy_seed(const void *f, float *lam_out, float *gF, const StepArgs &a,
                               cudaStream_t st) {
    AdjointArgs g{};
    for (int q = 0; q < Q; ++q) {
        g.lam_next[q] = nullptr;
        g.lam_out[q] = lam_out + q * a.g.pop;
    }
    g.gF = gF;
    const CellLaunch L = cell_launch(a.g);
    energy_seed_kernel<Q, T><<<L.grid, L.block, 0, st>>>(read_io<Q, T>(f, a.g), a, g);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_macro_seed(const void *f, const float *g_rho, const float *g_u,
                              float *lam_out, float *gF, const StepArgs &a, cudaStream_t st) {
    AdjointArgs g{};
    for (int q = 0; q < Q; ++q) {
        g.lam_next[q] = nullptr;
        g.lam_out[q] = lam_out + q * a.g.pop;
    }
    g.gF = gF;
    const CellLaunch L = cell_launch(a.g);
    macro_seed_kernel<Q, T><<<L.grid, L.block, 0, st>>>(read_io<Q, T>(f, a.g), a, g, g_rho, g_u);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_energy(const void *f, const StepArgs &a, double *part, cudaStream_t st) {
    const RedLaunch L = red_launch(a.g);
    energy_kernel<Q, T><<<L.blocks, L.block, 0, st>>>(read_io<Q, T>(f, a.g), a, part);
    return cudaGetLastError();
}

#define LBM_INSTANTIATE_ADJOINT(EXT, Q, T)                                                        \
    EXT template cudaError_t launch_adjoint<Q, T>(const void *, const float *, float *, float *, \
                                                  const StepArgs &, cudaStream_t);              \
    EXT template cudaError_t launch_energy_seed<Q, T>(const void *, float *, float *,            \
                                                      const StepArgs &, cudaStream_t);          \
    EXT template cudaError_t launch_macro_seed<Q, T>(const void *, const float *, const float *, \
                                                     float *, float *, const StepArgs &,        \
                                                     cudaStream_t);                             \
    EXT template cudaError_t launch_energy<Q, T>(const void *, const StepArgs &, double *,       \
                                                 cudaStream_t);

}  // namespace lbm
