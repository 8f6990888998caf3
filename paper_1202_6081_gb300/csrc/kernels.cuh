// Kernels of liblbm.so, templated over the lattice (Q = 27 or 15) and the
// storage type (float, __half, __nv_bfloat16).  kernels.cu instantiates the
// launchers; api.cu calls them.
#pragma once

#include "collide_q15.cuh"
#include "collide_q27.cuh"
#include "lattice.cuh"
#include "vec2.cuh"

#include <cstring>

namespace lbm {

struct StepArgs {
    Grid g;
    float w[27];           // relaxation rates omega_beta (first Q used)
    float F[3];            // uniform body force
    const float *Ffield;   // per-cell force [3][nz][ny][nx] or nullptr
    int has_force;         // 0: no force anywhere (the source term vanishes)
    int sr32;              // FP32 storage: incremental update, stochastically rounded
};

constexpr int kSMs = 152;

// Launch geometry shared by the per-cell kernels (cell_launch below).
struct CellLaunch {
    dim3 grid, block;
    // warps of the SM with the most blocks
    int sm_warps() const {
        const long long blocks = (long long)grid.x * grid.y * grid.z;
        return int((blocks + kSMs - 1) / kSMs * ((block.x * block.y + 31) / 32));
    }
};

// Blocks of at most 128 threads along x: rows of at least 17 threads take whole
// warps, a longer row blocks of equal width (192 threads: 96 + 96, not 128 + 64
// of 128: 384 x 128 x 192 D3Q27 FP16 195.6 -> 186.4 us a step, BF16 238 -> 227);
// shorter rows take the next power of two, so that a warp covers several rows
// instead of idling.
inline CellLaunch cell_launch(const Grid &g) {
    int bx;
    if (g.nx <= 16) {
        bx = 1;
        while (bx < g.nx) bx *= 2;
    } else {
        const int n = (g.nx + 127) / 128;
        bx = ((g.nx + n - 1) / n + 31) / 32 * 32;
    }
    int by = 128 / bx;
    if (by < 1) by = 1;
    CellLaunch L;
    L.block = dim3(bx, by, 1);
    L.grid = dim3((g.nx + bx - 1) / bx, (g.ny + by - 1) / by, g.nz);
    return L;
}

__device__ __forceinline__ bool cell_coords(const Grid &g, int &x, int &y, int &z) {
    x = blockIdx.x * blockDim.x + threadIdx.x;
    y = blockIdx.y * blockDim.y + threadIdx.y;
    z = blockIdx.z;
    return x < g.nx && y < g.ny;
}

__device__ __forceinline__ long long dense_index(const Grid &g, int x, int y, int z) {
    return ((long long)z * g.ny + y) * g.nx + x;
}

template <int Q>
struct Rates;
template <>
struct Rates<27> {
    using type = Rates27<float>;
};
template <>
struct Rates<15> {
    using type = Rates15<float>;
};

__device__ __forceinline__ Rates27<float> load_rates27(const StepArgs &a) {
    Rates27<float> r;
#pragma unroll
    for (int b = 0; b < 27; ++b) {
        r.w[b] = a.w[b];
        r.nw[b] = -a.w[b];
        r.omw[b] = 1.0f - a.w[b];
    }
    return r;
}

template <int Q>
__device__ __forceinline__ typename Rates<Q>::type load_rates(const StepArgs &a);
template <>
__device__ __forceinline__ Rates27<float> load_rates<27>(const StepArgs &a) {
    return load_rates27(a);
}
template <>
__device__ __forceinline__ Rates15<float> load_rates<15>(const StepArgs &a) {
    Rates15<float> r;
#pragma unroll
    for (int b = 0; b < 15; ++b) r.w[b] = a.w[b] * k15_inv(b);
    return r;
}

// The change d = f~ - f the collision makes (for the incremental update).
template <int Q>
__device__ __forceinline__ void collide_delta(const float (&f)[Q], float Fx, float Fy, float Fz,
                                              const typename Rates<Q>::type &r, bool has_force,
                                              float (&d)[Q]);
template <>
__device__ __forceinline__ void collide_delta<27>(const float (&f)[27], float Fx, float Fy,
                                                  float Fz, const Rates27<float> &r, bool,
                                                  float (&d)[27]) {
    collide27_delta(f, Fx, Fy, Fz, r, d);
}
template <>
__device__ __forceinline__ void collide_delta<15>(const float (&f)[15], float Fx, float Fy,
                                                  float Fz, const Rates15<float> &r,
                                                  bool has_force, float (&d)[15]) {
    collide15_delta(f, Fx, Fy, Fz, r, has_force, d);
}

template <int Q>
__device__ __forceinline__ void equilibrium(float drho, float ux, float uy, float uz, float Fx,
                                            float Fy, float Fz, float (&f)[Q]);
template <>
__device__ __forceinline__ void equilibrium<27>(float drho, float ux, float uy, float uz,
                                                float Fx, float Fy, float Fz, float (&f)[27]) {
    equilibrium27(drho, ux, uy, uz, Fx, Fy, Fz, f);
}
template <>
__device__ __forceinline__ void equilibrium<15>(float drho, float ux, float uy, float uz,
                                                float Fx, float Fy, float Fz, float (&f)[15]) {
    equilibrium15(drho, ux, uy, uz, Fx, Fy, Fz, f);
}

__device__ __forceinline__ void cell_force(const StepArgs &a, long long c, long long N, float &Fx,
                                           float &Fy, float &Fz) {
    if (a.Ffield) {
        Fx = __ldg(a.Ffield + c);
        Fy = __ldg(a.Ffield + N + c);
        Fz = __ldg(a.Ffield + 2 * N + c);
    } else {
        Fx = a.F[0];
        Fy = a.F[1];
        Fz = a.F[2];
    }
}

// Base pointer of every population plane of the source and destination
// buffers (plane alpha starts at buf + alpha * pop).  Passed by value, the
// table sits in the constant bank, so each access is one multiply-add of a
// 32-bit element offset onto a constant-bank base.
template <typename T>
struct StepIO {
    const T *in[27];
    T *out[27];
    const float4 *ref_in;  // momentum references of the input state (BF16), else unused
    float4 *ref_out;       // and of the output state
};

// Element e of a plane.  The offset is an unsigned 32-bit number of bytes, which
// the hardware adds to a uniform base in the access itself, where a signed
// element offset costs a 64-bit multiply-add per access on the FMA pipe (us a
// step: D3Q15 256^3 FP16 210 -> 201, BF16 229 -> 220; D3Q27 FP32 64^3 6.92 -> 6.76,
// 80^3 19.8 -> 18.6).  Planes of more than 2^32 bytes (FP32, over 2^30 elements) take
// the instantiations for ragged rows, which keep element offsets for FP32.
// kPlain: element offsets whatever the type, where those measured faster: the
// 16-bit D3Q27 step (256^3: FP16 327 against 338 us, BF16 391 against 398), whose
// registers are short, and some in-place kernels (kAAPlain).
template <bool kRag, bool kPlain = false, typename T>
__host__ __device__ __forceinline__ T *element(T *plane, int e) {
    using Byte = typename std::conditional<std::is_const<T>::value, const char, char>::type;
    if constexpr (kPlain || (kRag && sizeof(T) == 4))
        return plane + e;
    else
        return reinterpret_cast<T *>(reinterpret_cast<Byte *>(plane) +
                                     unsigned(e) * unsigned(sizeof(T)));
}
// 2-cell pair helpers for the packed kernel (x0 even, row pitch even).
template <typename T>
struct Pair;
// State loads: read-only, with an L2 prefetch-size hint of 256 bytes (the
// pulls stream through whole rows; measured +2.4 % FP16, +1.5 % BF16 at
// 512^3, FP32 unchanged).
__device__ __forceinline__ unsigned long long ld_nc_256_b64(const void *p) {
    unsigned long long v;
    asm("ld.global.nc.L2::256B.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ld_nc_256_b32(const void *p) {
    unsigned v;
    asm("ld.global.nc.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short ld_nc_256_b16(const void *p) {
    unsigned short v;
    asm("ld.global.nc.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
template <>
struct Pair<float> {
    __device__ __forceinline__ static f2 ld2(const float *p) { return f2(ld_nc_256_b64(p)); }
    __device__ __forceinline__ static float ld1(const float *p) {
        return __uint_as_float(ld_nc_256_b32(p));
    }
    __device__ __forceinline__ static void st2(float *p, f2 v) {
        __stcs(reinterpret_cast<float2 *>(p), make_float2(v.lo(), v.hi()));
    }
    // the step's stores (plain stores for FP32; see Pair16 for 16-bit)
    template <int q>
    __device__ __forceinline__ static void st2s(float *p, f2 v, unsigned) {
        st2(p, v);
    }
    template <int q>
    __device__ __forceinline__ static void st1x2s(float *plo, float *phi, f2 v, unsigned) {
        __stcs(plo, v.lo());
        __stcs(phi, v.hi());
    }
};
// 16-bit step stores: the pair is rounded together (pack_sr) and stored as one
// 32-bit word, or as two halves at separate addresses.
template <typename T>
struct Pair16 {
    template <int q>
    __device__ __forceinline__ static void st2s(T *p, f2 v, unsigned seed) {
        __stcs(reinterpret_cast<unsigned int *>(p), pack_sr<T, q>(v.lo(), v.hi(), seed));
    }
    template <int q>
    __device__ __forceinline__ static void st1x2s(T *plo, T *phi, f2 v, unsigned seed) {
        const unsigned d = pack_sr<T, q>(v.lo(), v.hi(), seed);
        __stcs(reinterpret_cast<unsigned short *>(plo), static_cast<unsigned short>(d & 0xffffu));
        __stcs(reinterpret_cast<unsigned short *>(phi), static_cast<unsigned short>(d >> 16));
    }
};
template <>
struct Pair<__half> : Pair16<__half> {
    __device__ __forceinline__ static f2 ld2(const __half *p) {
        const unsigned w = ld_nc_256_b32(p);
        const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(&w));
        return f2(v.x, v.y);
    }
    __device__ __forceinline__ static float ld1(const __half *p) {
        return __half2float(__ushort_as_half(ld_nc_256_b16(p)));
    }
};
template <>
struct Pair<__nv_bfloat16> : Pair16<__nv_bfloat16> {
    __device__ __forceinline__ static f2 ld2(const __nv_bfloat16 *p) {
        const unsigned w = ld_nc_256_b32(p);
        const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
        return f2(v.x, v.y);
    }
    __device__ __forceinline__ static float ld1(const __nv_bfloat16 *p) {
        return __bfloat162float(__ushort_as_bfloat16(ld_nc_256_b16(p)));
    }
};

// Seed of a thread's stochastic rounding (sr_seed) from four of its
// pre-collision values, of different directions, and its position.
template <int Q>
constexpr int kSeedPop = Q == 27 ? 11 : 9;
template <int Q>
__device__ __forceinline__ unsigned pair_seed(const f2 (&f)[Q], int own) {
    return sr_seed(f[1].v ^ f[6].v ^ f[kSeedPop<Q>].v ^ f[Q - 1].v, own);
}
// Which values the pair kernels hash: the pre-collision ones, or for D3Q15
// with FP16 storage the post-collision ones (either is a fixed function of
// the state; chosen by measurement: D3Q15 FP16 68.0k vs 62.4k MLUPS at 256^3
// hashing after the collision, D3Q15 BF16 61.5k vs 64.0k and D3Q27 the same
// or better before it).  The in-place kernels make the same choice, so that
// their states stay bit-identical to the two-buffer step's.
template <int Q, typename T>
constexpr bool kSeedAfterCollision = Q == 15 && Storage<T>::kScaled && !Storage<T>::kRef;

template <int Q>
__device__ __forceinline__ unsigned cell_seed(const float (&f)[Q], int own) {
    const unsigned a = __float_as_uint(f[1]) ^ __float_as_uint(f[6]);
    const unsigned b = __float_as_uint(f[kSeedPop<Q>]) ^ __float_as_uint(f[Q - 1]);
    return sr_seed(static_cast<unsigned long long>(b) << 32 | a, own);
}

// Relaxation rates pre-broadcast to both lanes, built on the host:
// D3Q27 omega, -omega, 1 - omega (divided by 216 for the kernels that fold
// the weights of 16-bit storage into their sums); D3Q15 omega / k_beta.
struct PackedRates {
    unsigned long long w[27], nw[27], omw[27];
    unsigned long long w15[15];
};

__device__ __forceinline__ Rates27<f2> load_rates_packed(const PackedRates &p) {
    Rates27<f2> r;
#pragma unroll
    for (int b = 0; b < 27; ++b) {
        r.w[b] = f2(p.w[b]);
        r.nw[b] = f2(p.nw[b]);
        r.omw[b] = f2(p.omw[b]);
    }
    return r;
}

// Factors of the two-cell kernels between stored values and the collision's
// values.  D3Q27 uses collide27_g: 16-bit inputs go in as stored (the
// weights are folded into its sums), and outputs carry G_i G_j G_k.
template <int Q, typename T>
__host__ __device__ constexpr bool kFoldedLoad() {
    return Q == 27 && Storage<T>::kScaled;
}
template <int Q, typename T>
__host__ __device__ constexpr float load_scale(int q) {
    return (Storage<T>::kScaled && Q != 27) ? float(weight<Q>(q)) : 1.0f;
}
template <int Q, typename T>
__host__ __device__ constexpr float store_scale(int q) {
    return float((Storage<T>::kScaled ? 1.0 / weight<Q>(q) : 1.0) / (Q == 27 ? g27(q) : 1));
}

// Row offsets (elements) of the 3 x 3 source rows of a pull, for cell row
// (y, z); wall[j][k] set where that source is beyond a bounce-back wall.
template <bool kWalls>
struct Rows {
    int off[3][3];
    bool wall[3][3];
    bool edge;  // some source is beyond a wall: the others take the plain loads
    int own;
};

template <bool kWalls>
__device__ __forceinline__ Rows<kWalls> pull_rows(const Grid &g, int y, int z) {
    Rows<kWalls> r;
    const int ys[3] = {(y + 1 == g.ny) ? 0 : y + 1, y, (y == 0) ? g.ny - 1 : y - 1};
    const int zs[3] = {(z + 1 == g.nz) ? 0 : z + 1, z, (z == 0) ? g.nz - 1 : z - 1};
    bool wy[3] = {false, false, false}, wz[3] = {false, false, false};
    if (kWalls) {
        wy[0] = (y + 1 == g.ny) && (g.bc & kWallY);
        wy[2] = (y == 0) && (g.bc & kWallY);
        wz[0] = (z + 1 == g.nz) && (g.bc & kWallZ);
        wz[2] = (z == 0) && (g.bc & kWallZ);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            r.off[j][k] = (zs[k] * g.ny + ys[j]) * g.px;
            r.wall[j][k] = kWalls && (wy[j] || wz[k]);
        }
    r.edge = wy[0] || wy[2] || wz[0] || wz[2];
    r.own = (z * g.ny + y) * g.px;
    return r;
}

// Cells a row's stores cover: the row rounded up to whole 32-byte sectors (the
// pitch has room).  A sector that is stored in part has to be filled from DRAM:
// D3Q27 FP32 at 126 x 117 x 133 cells took 76.2 us a step, at 128 (no partial
// sector) 64.9 us.  The threads past the row's end store there in the same
// instructions as the rest of their warp: the row's last cells again, in place what
// they make of the padding itself (PairCols), the adjoint step zeros (zero_padding).
template <typename T>
__host__ __device__ constexpr int stored_row(int nx) {
    constexpr int n = 32 / int(sizeof(T));
    return (nx + n - 1) / n * n;
}

// Columns of a thread's two cells (x0, x0 + 1), x0 even, and of their sources:
// xm left of x0, x1 (= x0 + 1 inside the row) right of x0, xp right of x0 + 1;
// at: where the thread stores.
// kRag: rows that do not fill their last sector.  The threads past the end
// (at >= nx) repeat the last pair.  In a row of odd length the last pair is one
// cell: its high lane reads in-range elements, is set to the low lane once the
// values are in registers (even_lanes) and stored in the row's padding.
// kApart (the in-place kernels, nx even): a thread past the end takes its two
// elements of the padding as a periodic row of their own, so that it reads and
// writes what no other thread does; the last pair's elements are overwritten by
// that pair's thread meanwhile.
template <bool kRag, bool kApart = false>
struct PairCols {
    int at, x0, xm, xp, nx;
    __host__ __device__ __forceinline__ PairCols(int x, int n) : at(x), x0(x), nx(n) {
        if (kRag && !kApart) x0 = last_pair();
        xm = (x0 == 0) ? nx - 1 : x0 - 1;
        xp = (kRag ? x0 + 2 >= nx : x0 + 2 == nx) ? 0 : x0 + 2;
        if (kRag && kApart && at >= nx) {
            xm = at + 1;
            xp = at;
        }
    }
    __host__ __device__ __forceinline__ bool single() const { return kRag && x0 + 1 == nx; }
    __host__ __device__ __forceinline__ int x1() const { return single() ? 0 : x0 + 1; }
    // whether the pair's cells are this thread's
    __host__ __device__ __forceinline__ bool owner() const { return !kRag || at < nx; }
    // the pair's column in a dense field, which has no padding
    __host__ __device__ __forceinline__ int field() const {
        return kRag && kApart ? last_pair() : x0;
    }
    // The same columns, in ragged rows from a value that the compiler cannot trace:
    // it would keep the addresses of the loads for the stores, and spill
    // (aa_odd_kernel D3Q27, periodic: 28-120 bytes, against none).
    __device__ __forceinline__ PairCols again() const {
        if constexpr (!kRag) return *this;
        int x = at;
        asm volatile("" : "+r"(x));
        return PairCols(x, nx);
    }

private:
    __host__ __device__ __forceinline__ int last_pair() const {
        return min(at, (nx - 1) & ~1);
    }
};

// End of the cells a row's threads store (T: the type stored).
template <typename T, bool kRag>
__host__ __device__ __forceinline__ int row_end(int nx) {
    return kRag ? stored_row<T>(nx) : nx;
}

template <int Q, bool kRag>
__device__ __forceinline__ void even_lanes(const PairCols<kRag> &X, f2 (&f)[Q]) {
    if constexpr (kRag) {
        if (X.single()) {
#pragma unroll
            for (int q = 0; q < Q; ++q) f[q] = f2(f[q].lo(), f[q].lo());
        }
    }
}

// Zeros in the lanes that a thread stores in its row's padding.
template <int Q, bool kRag>
__device__ __forceinline__ void zero_padding(const PairCols<kRag> &X, f2 (&f)[Q]) {
    if constexpr (kRag) {
        if (X.single() || !X.owner()) {
#pragma unroll
            for (int q = 0; q < Q; ++q) f[q] = f2(X.owner() ? f[q].lo() : 0.0f, 0.0f);
        }
    }
}

// BF16 momentum references (see lattice.cuh) for the pair kernels.
//
// Reader: adds to the pulled raw values f[q] of cells (x0, x0 + 1) the
// reference of each value's producer: for e_x = 0 both from the pair of the
// source row, for e_x = +1 from the pairs of x0 - 1 and x0, for e_x = -1 of
// x0 + 1 and x0 + 2; behind a wall minus that of the own pair.  A source row
// (e_y, e_z) needs two components of J at most, loaded narrow to keep
// registers free: the row e_y = e_z = 0 only Jx (axis populations), rows
// with e_z = 0 (Jx, Jy), rows with e_y = 0 (Jz, Jx) -- J is stored as
// (Jx, Jy, Jz, Jx) so that both pairs are aligned 8-byte loads -- and the
// rows with e_y, e_z both nonzero (Jy, Jz), only of the own column (their
// corners carry no reference).
template <int ey, int ez>
__device__ __forceinline__ float4 load_ref(const float4 *p) {
    if constexpr (ey == 0 && ez == 0) {
        return make_float4(__ldg(&p->x), 0.0f, 0.0f, 0.0f);
    } else if constexpr (ez == 0) {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
        return make_float4(v.x, v.y, 0.0f, 0.0f);
    } else if constexpr (ey == 0) {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(p) + 1);
        return make_float4(v.y, 0.0f, v.x, 0.0f);
    } else {
        return __ldg(p);
    }
}

// kSel: with the wall selects.
template <int Q, bool kSel, bool kWalls, bool kRag, bool kApart>
__device__ __forceinline__ void add_refs_pair(const float4 *__restrict__ ref, const Rows<kWalls> &R,
                                              const PairCols<kRag, kApart> &X, f2 (&f)[Q]) {
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        if constexpr (has_ref<Q>(q)) {
            constexpr int i = ex<Q>(q), j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
            constexpr int cy = ey<Q>(q), cz = ez<Q>(q);
            float rlo, rhi;
            if (kSel && R.wall[j][k]) {
                rlo = rhi = -ref_dot<Q, q>(load_ref<cy, cz>(ref + ((R.own + X.x0) >> 1)));
            } else {
                const float4 *row = ref + (R.off[j][k] >> 1);
                const float4 C = load_ref<cy, cz>(row + (X.x0 >> 1));
                if constexpr (i == 0) {
                    rlo = rhi = ref_dot<Q, q>(C);
                } else if constexpr (i == 1) {
                    rlo = ref_dot<Q, q>(load_ref<cy, cz>(row + (X.xm >> 1)));
                    rhi = ref_dot<Q, q>(C);
                } else {
                    rlo = ref_dot<Q, q>(kRag ? load_ref<cy, cz>(row + (X.x1() >> 1)) : C);
                    rhi = ref_dot<Q, q>(load_ref<cy, cz>(row + (X.xp >> 1)));
                }
            }
            f[q] = f[q] + f2(rlo, rhi);
        }
    });
}

// Writer: the pair's reference J = 3 u-bar (mean velocity of the two cells).
__device__ __forceinline__ float4 pair_ref(f2 ux, f2 uy, f2 uz) {
    const float jx = 1.5f * (ux.lo() + ux.hi());
    return make_float4(jx, 1.5f * (uy.lo() + uy.hi()), 1.5f * (uz.lo() + uz.hi()), jx);
}

// Stored value of population q of a pair from its post-collision value v
// times the store scale sc: v sc, minus e_q . J for the referenced
// populations of BF16 storage.
template <int Q, typename T, int q>
__device__ __forceinline__ f2 stored_pair(f2 v, float sc, const float4 &J) {
    if constexpr (Storage<T>::kRef && has_ref<Q>(q))
        return vfma(v, f2(sc), f2(-ref_dot<Q, q>(J)));
    else
        return sc == 1.0f ? v : v * f2(sc);
}

// ---- one cell's distributions, for the kernels that read or load a state ----
//
// These kernels move a state once and compute little, so each access has to be
// cheap: plane base pointers from the constant bank plus one 32-bit offset per
// population (as in the step kernels), and the common case -- two-buffer
// layout, no walls -- without the layout and wall selects.

// Population q's stored value -> deviation f - w; prod: the cell whose collision
// produced it (the momentum reference of BF16 storage).
template <int Q, typename T, int q>
__device__ __forceinline__ float load_cell(const T *at, const float4 *ref, int prod, bool wall) {
    float v = Pair<T>::ld1(at);
    if constexpr (Storage<T>::kRef && has_ref<Q>(q)) {
        const float r = ref_dot<Q, q>(load_ref<ey<Q>(q), ez<Q>(q)>(ref + (prod >> 1)));
        v += wall ? -r : r;
    }
    return Storage<T>::kScaled ? v * float(weight<Q>(q)) : v;
}

// Pre-collision deviations f_alpha(x) - w_alpha of one cell (slot order).
template <int Q, typename T>
__device__ __forceinline__ void gather(const StepIO<T> &io, const Grid &g, int x, int y, int z,
                                       float (&f)[Q]) {
    const int xs[3] = {(x + 1 == g.nx) ? 0 : x + 1, x, (x == 0) ? g.nx - 1 : x - 1};
    if (g.layout == kPull && g.bc == 0) {
        const Rows<false> R = pull_rows<false>(g, y, z);
        static_for<Q>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            const int src = R.off[ey<Q>(q) + 1][ez<Q>(q) + 1] + xs[ex<Q>(q) + 1];
            f[q] = load_cell<Q, T, q>(io.in[q] + src, io.ref_in, src, false);
        });
        return;
    }
    const Rows<true> R = pull_rows<true>(g, y, z);
    const int own = R.own + x;
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr int i = ex<Q>(q) + 1, j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
        const bool wall = R.wall[j][k];
        const int prod = wall ? own : R.off[j][k] + xs[i];
        const bool opp = g.layout == kPull ? wall : g.layout == kAASwapped && !wall;
        const T *plane = opp ? io.in[opposite<Q>(q)] : io.in[q];
        f[q] = load_cell<Q, T, q>(plane + (g.layout == kAANatural ? own : prod), io.ref_in, prod,
                                  wall);
    });
}

// Inverse of the pull: place the pre-collision values f_alpha(x) of one cell
// where the next step will read them (the AA scheme loads into its natural
// layout).  With momentum references (BF16) io.ref_out must already hold J of
// every pair (ref_init_kernel), and each value is stored relative to the
// reference of its producer, as a reader will add it back.
template <int Q, typename T>
__device__ __forceinline__ void scatter_state(const StepIO<T> &io, const Grid &g, int x, int y,
                                              int z, const float (&f)[Q]) {
    const int xs[3] = {(x + 1 == g.nx) ? 0 : x + 1, x, (x == 0) ? g.nx - 1 : x - 1};
    const Rows<true> R = pull_rows<true>(g, y, z);
    const int own = R.own + x;
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr int i = ex<Q>(q) + 1, j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
        const bool wall = R.wall[j][k];
        const int prod = wall ? own : R.off[j][k] + xs[i];
        float ref = 0.0f;
        if constexpr (Storage<T>::kRef && has_ref<Q>(q)) {
            const float r = ref_dot<Q, q>(load_ref<ey<Q>(q), ez<Q>(q)>(io.ref_out + (prod >> 1)));
            ref = wall ? -r : r;
        }
        // opposite slots have equal weights
        T *plane = g.layout == kPull && wall ? io.out[opposite<Q>(q)] : io.out[q];
        store_dev<Q, T>(plane + (g.layout == kPull ? prod : own), q, f[q], ref);
    });
}

// FP64 arithmetic of the state readers and writers, on the integer pipe.  GB300
// issues about one FP64 operation per clock and SM (64-bit integer conversions
// too), so one FP64 addition per population takes longer than the memory
// traffic: 192^3 D3Q27 FP32, get_state 709 us and set_state 668 us with the
// FP64 pipe 86-89 % busy, against 338 us of bytes.  The functions below return
// the same bits; values outside their range take the FP64 instruction.

// float -> double, exactly.
__device__ __forceinline__ double widen(float v) {
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u || m == 0u)  // normal or zero
        return __hiloint2double(int((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)),
                                int(b << 29));
    return double(v);
}

// exponent of a weight: 2^e <= w < 2^(e + 1), and its mantissa w 2^(52 - e)
__host__ __device__ constexpr int weight_exponent(double w) {
    int e = 0;
    while (w < 1.0) {
        w *= 2.0;
        --e;
    }
    return e;
}
__host__ __device__ constexpr long long weight_mantissa(double w) {
    for (int i = weight_exponent(w); i < 52; ++i) w *= 2.0;
    return (long long)w;
}

// w_q + v, rounded to nearest even.  In units of 2^(e - 52) both are integers
// (|v| >= 2^(e - 29): 24 significant bits), their sum s is exact, and one of
// three positions of its leading bit gives the result; only the highest one
// drops a bit.  |v| < 2^(e - 54), zero included, leaves w.
template <int Q, int q>
__device__ __forceinline__ double weight_plus(float v) {
    constexpr double w = weight<Q>(q);
    constexpr int e = weight_exponent(w);
    constexpr long long mw = weight_mantissa(w);
    const unsigned b = __float_as_uint(v);
    const int up = int(b >> 23 & 0xffu) - (127 + e - 29);
    if (up < -25) return w;
    if (up >= 0 && up <= 30) {
        const long long m = (long long)((b & 0x7fffffu) | 0x800000u) << up;
        const unsigned long long s = (unsigned long long)(int(b) < 0 ? mw - m : mw + m);
        const unsigned top = unsigned(s >> 51);
        if (top - 1u < 7u) {  // 2^51 <= s < 2^54
            unsigned long long r = s;
            int er = e;
            if (top == 1u) {
                r = s << 1;
                er = e - 1;
            } else if (top >= 4u) {
                r = (s + (s >> 1 & 1u)) >> 1;
                er = e + 1;
            }
            return __longlong_as_double((long long)r + ((long long)(1022 + er) << 52));
        }
    }
    return w + double(v);
}

// float(f - w_q): the exact difference, rounded once to nearest even.  For f in
// w's binade or a neighbouring one both are integers in units of 2^(e - 53), and
// a difference below 2^53 is what the FP64 subtraction gives exactly.  It is
// shifted into 32 bits, what falls off kept as a sticky bit, and converted.
template <int Q, int q>
__device__ __forceinline__ float deviation(double f) {
    constexpr double w = weight<Q>(q);
    constexpr int e = weight_exponent(w);
    constexpr long long mw = 2 * weight_mantissa(w);
    const unsigned hi = unsigned(__double2hiint(f));
    const unsigned up = (hi >> 20) - unsigned(1023 + e - 1);
    if (up <= 2u) {
        const unsigned long long m =
            (unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | unsigned(__double2loint(f));
        const long long d = (long long)(m << up) - mw;
        const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
        const unsigned ah = unsigned(a >> 32), al = unsigned(a);
        if (ah < 1u << 21) {
            const int n = 32 - __clz(int(ah));
            unsigned t = __funnelshift_r(al, ah, n);
            if (al & ((1u << n) - 1u)) t |= 1u;
            const float r = __uint2float_rn(t) * __uint_as_float(unsigned(127 + e - 53 + n) << 23);
            return d < 0 ? -r : r;
        }
    }
    return float(f - w);
}

// One cell's pulled populations, as deviations f - w.
// kRag: see element().
template <int Q, typename T, bool kRag, bool kWalls>
__device__ __forceinline__ void pull_cell(const StepIO<T> &io, const Rows<kWalls> &R, int x,
                                          int nx, float (&f)[Q]) {
    const int xs[3] = {(x + 1 == nx) ? 0 : x + 1, x, (x == 0) ? nx - 1 : x - 1};
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr int i = ex<Q>(q) + 1, j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
        const bool wall = kWalls && R.wall[j][k];
        const int src = wall ? R.own + x : R.off[j][k] + xs[i];
        const T *at = element<kRag>(wall ? io.in[opposite<Q>(q)] : io.in[q], src);
        f[q] = load_cell<Q, T, q>(at, io.ref_in, src, wall);
    });
}

// One fused step, one cell per thread, for small grids with rows of odd length.
// A small grid does not fill the chip and its step takes as long as
// one thread's chain of instructions, which is shorter here.  (Scalar
// arithmetic rounds differently from the packed one, so grids that can also run
// in place, with even rows, keep the two-cell kernel at every size: their
// states are the same bit for bit in either scheme.)  See kOneCellWarps.
// BF16 storage: the cells x (even) and x + 1, in neighbouring lanes, exchange their
// velocities for the pair's reference, so every lane takes part: lanes beyond the
// grid work on a clamped cell and store nothing.
template <int Q, typename T, bool kWalls, bool kForm>
__global__ void __launch_bounds__(128) step1_kernel(const StepIO<T> io, const StepArgs a) {
    int x, y, z;
    const bool inside = cell_coords(a.g, x, y, z);
    if constexpr (Storage<T>::kRef) {
        x = min(x, a.g.nx - 1);
        y = min(y, a.g.ny - 1);
    } else {
        if (!inside) return;
    }
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    float f[Q];
    pull_cell<Q, T, false>(io, R, x, a.g.nx, f);
    unsigned seed = 0;
    if constexpr (Storage<T>::kScaled) seed = cell_seed<Q>(f, R.own + x);
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    float Fx = 0.0f, Fy = 0.0f, Fz = 0.0f, ux, uy, uz;
    if (Q == 27 || kForm) cell_force(a, dense_index(a.g, x, y, z), N, Fx, Fy, Fz);
    const typename Rates<Q>::type r = load_rates<Q>(a);
    // the rate-1 form between walls only: periodic, the general one schedules better
    // (9^3: 2.20 / 2.39 us; walled 2.59 / 2.27); BF16 2.76 / 3.90 at 17^3 walled
    constexpr bool kRateOne = Q == 27 && kForm && kWalls && !Storage<T>::kRef;
    if constexpr (kRateOne)
        collide27_g<float, false, true>(f, Fx, Fy, Fz, r, ux, uy, uz);
    else if constexpr (Q == 27)
        collide27<float>(f, Fx, Fy, Fz, r, ux, uy, uz);
    else
        collide15<float>(f, Fx, Fy, Fz, r, kForm, ux, uy, uz);
    float4 J = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if constexpr (Storage<T>::kRef) {
        const float px = __shfl_xor_sync(0xffffffffu, ux, 1);
        const float py = __shfl_xor_sync(0xffffffffu, uy, 1);
        const float pz = __shfl_xor_sync(0xffffffffu, uz, 1);
        if ((x ^ 1) < a.g.nx)  // both cells of the pair exist (a + b == b + a exactly)
            J = make_float4(1.5f * (ux + px), 1.5f * (uy + py), 1.5f * (uz + pz), 0.0f);
        else
            J = make_float4(3.0f * ux, 3.0f * uy, 3.0f * uz, 0.0f);
        J.w = J.x;
        if (!inside) return;
        if ((x & 1) == 0) __stcs(io.ref_out + ((R.own + x) >> 1), J);
    }
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr float scale = kRateOne ? store_scale<Q, float>(q) : 1.0f;
        T *at = element<false>(io.out[q], R.own + x);
        if constexpr (Storage<T>::kScaled) {
            float ref = 0.0f;
            if constexpr (Storage<T>::kRef && has_ref<Q>(q)) ref = ref_dot<Q, q>(J);
            const float v = fmaf(f[q], scale * float(1.0 / weight<Q>(q)), -ref);
            __stcs(reinterpret_cast<unsigned short *>(at),
                   static_cast<unsigned short>(pack_sr<T, q>(v, 0.0f, seed) & 0xffffu));
        } else {
            __stcs(at, scale == 1.0f ? f[q] : f[q] * scale);
        }
    });
}

// One fused step with the stochastically rounded FP32 update (LBM_F32_SR), one
// cell per thread: the update is f~ = f + d with d the collision's change, and
// that last addition is rounded stochastically (add_sr32), so that no rounding
// error repeats identically step after step at a steady state.
template <int Q, bool kWalls>
__global__ void __launch_bounds__(128) step_sr32_kernel(const StepIO<float> io, const StepArgs a) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    float f[Q];
    pull_cell<Q, float, true>(io, R, x, a.g.nx, f);
    const unsigned seed = cell_seed<Q>(f, R.own + x);
    float Fx, Fy, Fz;
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    cell_force(a, dense_index(a.g, x, y, z), N, Fx, Fy, Fz);
    const typename Rates<Q>::type r = load_rates<Q>(a);
    float d[Q];
    collide_delta<Q>(f, Fx, Fy, Fz, r, a.has_force != 0, d);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        __stcs(io.out[q] + (R.own + x), add_sr32(f[q], d[q], sr_bits<q>(seed)));
    });
}

// The values of a plane's row (offset of its start) at x0 - i and x0 + 1 - i.
// kRowFirst: the row's pointer, then the column (see kAAPlain).
template <bool kPlain = false, bool kRowFirst = false, typename T, bool kRag, bool kApart>
__device__ __forceinline__ f2 ld_shifted(const T *plane, int row, int i,
                                         const PairCols<kRag, kApart> &X) {
    if constexpr (kRowFirst) {
        plane += row;
        row = 0;
    }
    const T *own = element<kRag, kPlain>(plane, row + X.x0);
    if (i == 0) return Pair<T>::ld2(own);
    if (i == 1)
        return f2(Pair<T>::ld1(element<kRag, kPlain>(plane, row + X.xm)), Pair<T>::ld1(own));
    return f2(Pair<T>::ld1(kRag ? element<kRag, kPlain>(plane, row + X.x1()) : own + 1),
              Pair<T>::ld1(element<kRag, kPlain>(plane, row + X.xp)));
}

// Pair gather: population q of cells (x0, x0 + 1) from the pull sources.
template <int Q, typename T>
constexpr bool kStepPlain = Q == 27 && Storage<T>::kScaled;

template <int Q, typename T, bool kSel, bool kWalls, bool kRag>
__device__ __forceinline__ f2 pull_pair(const StepIO<T> &io, const Rows<kWalls> &R, int q,
                                        const PairCols<kRag> &X) {
    const int i = ex<Q>(q), j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
    if (kSel && R.wall[j][k])
        return Pair<T>::ld2(
            element<kRag, kStepPlain<Q, T>>(io.in[opposite<Q>(q)], R.own + X.x0));
    return ld_shifted<kStepPlain<Q, T>>(io.in[q], R.off[j][k], i, X);
}

// All populations of the pair as stored, BF16 references added.  The wall
// selects are compiled beside the plain loads and taken by the rows along a
// wall only: with selects everywhere the 128 x 117 x 133 step took 69.5 us
// between walls against 64.9 us periodic.
// kShort: rows of less than a warp, where one warp holds rows of both kinds and
// would run both: the selects alone.
template <int Q, typename T, bool kShort = false, bool kWalls, bool kRag>
__device__ __forceinline__ void pull_pairs(const StepIO<T> &io, const Rows<kWalls> &R,
                                           const PairCols<kRag> &X, f2 (&f)[Q]) {
    const auto pull = [&](auto sel) {
        constexpr bool kSel = decltype(sel)::value;
        static_for<Q>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            f[q] = pull_pair<Q, T, kSel>(io, R, q, X);
        });
        if constexpr (Storage<T>::kRef) add_refs_pair<Q, kSel>(io.ref_in, R, X, f);
    };
    if constexpr (kShort) {
        pull(std::integral_constant<bool, kWalls>{});
    } else {
        if (kWalls && (R.edge || blockDim.x < 32))
            pull(std::integral_constant<bool, kWalls>{});
        else
            pull(std::false_type{});
    }
    even_lanes(X, f);
}

// Body force of the pair (x0, x0 + 1): the field (4-byte alignment only is
// required of it: single loads), else the uniform force.
template <bool kRag, bool kApart>
__device__ __forceinline__ void pair_force(const StepArgs &a, const PairCols<kRag, kApart> &X,
                                           int y, int z, f2 &Fx, f2 &Fy, f2 &Fz) {
    if (a.Ffield) {
        const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
        const float *p = a.Ffield + dense_index(a.g, X.field(), y, z);
        const int n = X.single() ? 0 : 1;
        Fx = f2(__ldg(p), __ldg(p + n));
        Fy = f2(__ldg(p + N), __ldg(p + N + n));
        Fz = f2(__ldg(p + 2 * N), __ldg(p + 2 * N + n));
    } else {
        Fx = f2(a.F[0]);
        Fy = f2(a.F[1]);
        Fz = f2(a.F[2]);
    }
}

// One fused D3Q27 step, two neighbouring cells (x0, x0 + 1) per thread with
// the collision in packed f32x2 arithmetic.  Loads of
// populations with e_x = 0 and all stores are aligned 2-element accesses;
// e_x = +-1 sources are two single loads (x0 - 1, x0) or (x0 + 1, x0 + 2).
// Blocks of 128 per SM, by measurement (us a step at 256^3): FP32 storage 5 (518;
// 6: 523).  FP16 6 (327 / 326 / 323 at 6 / 5 / 7 blocks at the rate-1 form, at
// 512^3 2642 / 2653 at 6 / 7; general rates 372 / 392 at 6 / 7).  BF16 with its
// reference loads 5 (388.6 / 391.8 / 414 at 5 / 6 / 7; 32^3 2.91 / 3.10 at 5 / 6),
// with the wall selects 6 (401 / 426 at 6 / 5).
template <typename T, bool kWalls>
constexpr int kStep2Blocks = Storage<T>::kScaled && (kWalls || !Storage<T>::kRef) ? 6 : 5;

// kEq: the rates from the trace on are all 1 (relax27).
// kShort: see pull_pairs.
template <typename T, bool kWalls, bool kEq, bool kRag, bool kShort = false>
__global__ void __launch_bounds__(128, (kStep2Blocks<T, kWalls>))
    step2_kernel(const StepIO<T> io, const StepArgs a, const PackedRates pr) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (2 * t >= row_end<T, kRag>(a.g.nx) || y >= a.g.ny) return;
    const PairCols<kRag> X(2 * t, a.g.nx);
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    f2 f[27];  // weight-scaled 16-bit values go in as stored (collide27_g)
    pull_pairs<27, T, kShort>(io, R, X, f);
    const int own = R.own + X.x0;
    const unsigned seed = pair_seed<27>(f, own);
    f2 Fx, Fy, Fz;
    pair_force(a, X, y, z, Fx, Fy, Fz);
    const Rates27<f2> r = load_rates_packed(pr);
    f2 ux, uy, uz;
    collide27_g<f2, Storage<T>::kScaled, kEq>(f, Fx, Fy, Fz, r, ux, uy, uz);
    float4 J = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if constexpr (Storage<T>::kRef) {
        J = pair_ref(ux, uy, uz);
        __stcs(io.ref_out + ((R.own + X.at) >> 1), J);
    }
    static_for<27>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        const f2 v = stored_pair<27, T, q>(f[q], store_scale<27, T>(q), J);
        Pair<T>::template st2s<q>(element<kRag, kStepPlain<27, T>>(io.out[q], R.own + X.at), v,
                                  seed);
    });
}

// One fused D3Q15 step, two neighbouring cells per thread in packed f32x2
// arithmetic; loads and stores as in step2_kernel.
// kForce = false (no force anywhere) compiles the force-free cascade alone:
// without the forced path beside it the kernel needs fewer registers (no
// spills at 5 blocks per SM with 16-bit storage, against 104-128 bytes;
// FP16 77.2k against 70.7k MLUPS at 256^3).  Blocks per SM, by measurement at
// 256^3 (us a step): 16-bit 6 without force (BF16 220 / 222 / 227 at 6 / 5 / 7,
// walled FP16 198 / 212 / 204), FP16 without walls 7 (196.6 / 201.7 at 7 / 6; in
// ragged rows 53.3 / 51.2 at 250 x 128 x 128), 5 with it (FP16 245 / 262 / 257 at
// 5 / 4 / 6); FP32 storage 4 (no spills; without force its 94 registers admit 5).
template <typename T, bool kWalls, bool kForce, bool kRag>
constexpr int kQ15Blocks = !Storage<T>::kScaled                           ? 4
                           : kForce                                       ? 5
                           : kWalls || kRag || Storage<T>::kRef           ? 6
                                                                          : 7;

template <typename T, bool kWalls, bool kForce, bool kRag, bool kShort = false>
__global__ void __launch_bounds__(128, (kQ15Blocks<T, kWalls, kForce, kRag>))
    step2_q15_kernel(const StepIO<T> io, const StepArgs a, const PackedRates pr) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (2 * t >= row_end<T, kRag>(a.g.nx) || y >= a.g.ny) return;
    const PairCols<kRag> X(2 * t, a.g.nx);
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    const int own = R.own + X.x0;
    f2 f[15];
    pull_pairs<15, T, kShort>(io, R, X, f);
    if constexpr (Storage<T>::kScaled) {
        static_for<15>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            f[q] = f[q] * f2(float(weight<15>(q)));
        });
    }
    unsigned seed = 0;
    if constexpr (!kSeedAfterCollision<15, T>) seed = pair_seed<15>(f, own);
    f2 Fx = f2(0.0f), Fy = f2(0.0f), Fz = f2(0.0f);
    if constexpr (kForce) pair_force(a, X, y, z, Fx, Fy, Fz);
    Rates15<f2> r;
#pragma unroll
    for (int b = 0; b < 15; ++b) r.w[b] = f2(pr.w15[b]);
    f2 ux, uy, uz;
    collide15<f2>(f, Fx, Fy, Fz, r, kForce, ux, uy, uz);
    float4 J = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if constexpr (Storage<T>::kRef) {
        J = pair_ref(ux, uy, uz);
        __stcs(io.ref_out + ((R.own + X.at) >> 1), J);
    }
    if constexpr (kSeedAfterCollision<15, T>) seed = pair_seed<15>(f, own);
    static_for<15>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        const f2 v = stored_pair<15, T, q>(f[q], store_scale<15, T>(q), J);
        Pair<T>::template st2s<q>(element<kRag, kStepPlain<15, T>>(io.out[q], R.own + X.at), v,
                                  seed);
    });
}

// ---- in-place (AA) streaming: one buffer, two kinds of step -------------
//
// Even step (layout kAANatural -> kAASwapped): each cell reads its own
// populations f_a(x) from slot a, collides, and writes f~_a(x) back to its
// own cell, slot opp(a).  Odd step (kAASwapped -> kAANatural): each cell
// reads f_a(x) = f~_a(x - e_a) from slot opp(a) of its upstream neighbour (or
// from its own slot a behind a bounce-back wall), collides, and writes
// f~_a(x) to slot a of its downstream neighbour x + e_a (or to its own slot
// opp(a) when x + e_a is behind a wall), where the next even step reads it.
// In both steps a thread reads and writes the same set of locations, so the
// update is race-free in place.  Both use two cells per thread (nx even).

template <int Q>
struct PairCollide;
// kForce = false: no force anywhere (D3Q15 then takes the force-free
// cascade; the D3Q27 collision takes any force, zero included, the same way).
template <>
struct PairCollide<27> {
    template <bool kWeighted, bool kEq, bool>
    __device__ __forceinline__ static void run(f2 (&f)[27], f2 Fx, f2 Fy, f2 Fz,
                                               const PackedRates &pr, f2 &ux, f2 &uy, f2 &uz) {
        const Rates27<f2> r = load_rates_packed(pr);
        collide27_g<f2, kWeighted, kEq>(f, Fx, Fy, Fz, r, ux, uy, uz);
    }
};
template <>
struct PairCollide<15> {
    template <bool, bool, bool kForce>
    __device__ __forceinline__ static void run(f2 (&f)[15], f2 Fx, f2 Fy, f2 Fz,
                                               const PackedRates &pr, f2 &ux, f2 &uy, f2 &uz) {
        Rates15<f2> r;
#pragma unroll
        for (int b = 0; b < 15; ++b) r.w[b] = f2(pr.w15[b]);
        collide15<f2>(f, Fx, Fy, Fz, r, kForce, ux, uy, uz);
    }
};

// Raw pulled values -> the collision's inputs: BF16 references added (their
// producers are the pull sources, see lattice.cuh), then the load scale.
template <int Q, typename T, bool kWalls, bool kRag>
__device__ __forceinline__ void pair_inputs(const StepIO<T> &io, const Rows<kWalls> &R,
                                            const PairCols<kRag, true> &X, f2 (&f)[Q]) {
    if constexpr (Storage<T>::kRef) add_refs_pair<Q, kWalls>(io.ref_in, R, X, f);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        constexpr float sc = load_scale<Q, T>(q);
        if constexpr (sc != 1.0f) f[q] = f[q] * f2(sc);
    });
}

// The collision of an in-place step, then the pair's reference (BF16).
template <int Q, typename T, bool kEq, bool kForce, bool kRag>
__device__ __forceinline__ float4 pair_collide(const StepIO<T> &io, const StepArgs &a,
                                               const PackedRates &pr,
                                               const PairCols<kRag, true> &X, int y, int z,
                                               int own, f2 (&f)[Q]) {
    f2 Fx = f2(0.0f), Fy = f2(0.0f), Fz = f2(0.0f), ux, uy, uz;
    if constexpr (kForce) pair_force(a, X, y, z, Fx, Fy, Fz);
    PairCollide<Q>::template run<kFoldedLoad<Q, T>(), kEq, kForce>(f, Fx, Fy, Fz, pr, ux, uy, uz);
    float4 J = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if constexpr (Storage<T>::kRef) {
        J = pair_ref(ux, uy, uz);
        __stcs(io.ref_out + (own >> 1), J);
    }
    return J;
}

// Element offsets instead of byte offsets (element()) where those measured slower
// in the in-place kernels: 256^3 us a step, bytes / elements, D3Q27 BF16 466 / 411
// (452 with row and column summed first), FP32 at general rates 545 / 527 (598);
// ragged rows (250 x 256 x 256) D3Q27 FP16 between walls 348 / 339 (340), though
// periodic 319 / 329 and D3Q15 FP16 200 / 214; else bytes: D3Q27 FP16 320 / 353,
// D3Q15 FP16 204 / 231.
template <int Q, typename T, bool kEq, bool kRag>
constexpr bool kAAPlain = kRag || (Q == 27 && (Storage<T>::kRef || (sizeof(T) == 4 && !kEq)));

template <int Q, typename T, bool kWalls, bool kEq, bool kForce, bool kRag>
__global__ void __launch_bounds__(128) aa_even_kernel(const StepIO<T> io, const StepArgs a,
                                                      const PackedRates pr) {
    constexpr bool kPlain = kAAPlain<Q, T, kEq, kRag>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (2 * t >= row_end<T, kRag>(a.g.nx) || y >= a.g.ny) return;
    const PairCols<kRag, true> X(2 * t, a.g.nx);
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);  // producers of the values (BF16)
    const int own = R.own + X.at;
    f2 f[Q];
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        f[q] = Pair<T>::ld2(element<kRag, kPlain>(io.in[q], own));
    });
    pair_inputs<Q, T>(io, R, X, f);
    unsigned seed = 0;
    if constexpr (!kSeedAfterCollision<Q, T>) seed = pair_seed<Q>(f, own);
    const float4 J = pair_collide<Q, T, kEq, kForce>(io, a, pr, X, y, z, own, f);
    if constexpr (kSeedAfterCollision<Q, T>) seed = pair_seed<Q>(f, own);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        const f2 v = stored_pair<Q, T, q>(f[q], store_scale<Q, T>(q), J);
        Pair<T>::template st2s<q>(element<kRag, kPlain>(io.out[opposite<Q>(q)], own), v, seed);
    });
}

// Blocks of 128 per SM, from measurement: D3Q27 at 5 (96 registers; FP32
// storage without spills, 16-bit with 40 bytes: 38.3k vs 33.3k MLUPS FP16 at
// 512^3 against 3 blocks); D3Q15 with force at 4 (8-48 bytes of spills),
// without force at 5 (no spills; FP16 77.7k vs 68.9k MLUPS at 256^3 against 4).
template <int Q, typename T, bool kForce>
constexpr int kAAOddBlocks = Q == 27 ? 5 : (kForce ? 4 : 5);

template <int Q, typename T, bool kWalls, bool kEq, bool kForce, bool kRag>
__global__ void __launch_bounds__(128, (kAAOddBlocks<Q, T, kForce>))
    aa_odd_kernel(const StepIO<T> io, const StepArgs a, const PackedRates pr) {
    constexpr bool kPlain = kAAPlain<Q, T, kEq, kRag>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (2 * t >= row_end<T, kRag>(a.g.nx) || y >= a.g.ny) return;
    const PairCols<kRag, true> X(2 * t, a.g.nx);
    const Rows<kWalls> R = pull_rows<kWalls>(a.g, y, z);
    const int own = R.own + X.at;
    // rows along a wall take the wall selects, the others the plain accesses
    // (see pull_pairs)
    const bool edge = kWalls && (R.edge || blockDim.x < 32);
    f2 f[Q];
    const auto load = [&](auto sel) {
        static_for<Q>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            constexpr int i = ex<Q>(q), j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
            if (decltype(sel)::value && R.wall[j][k])
                f[q] = Pair<T>::ld2(element<kRag, kPlain>(io.in[q], own));
            else
                f[q] = ld_shifted<kPlain, kPlain && !kRag>(io.in[opposite<Q>(q)], R.off[j][k], i,
                                                          X);
        });
    };
    if (edge)
        load(std::integral_constant<bool, kWalls>{});
    else
        load(std::false_type{});
    pair_inputs<Q, T>(io, R, X, f);
    unsigned seed = 0;
    if constexpr (!kSeedAfterCollision<Q, T>) seed = pair_seed<Q>(f, own);
    const float4 J = pair_collide<Q, T, kEq, kForce>(io, a, pr, X, y, z, own, f);
    if constexpr (kSeedAfterCollision<Q, T>) seed = pair_seed<Q>(f, own);
    const PairCols<kRag, true> Y = X.again();
    const auto store = [&](auto sel) {
        static_for<Q>([&](auto iq) {
            constexpr int q = decltype(iq)::value;
            constexpr int i = ex<Q>(q), j = ey<Q>(q) + 1, k = ez<Q>(q) + 1;
            constexpr int o = opposite<Q>(q);
            const f2 v = stored_pair<Q, T, q>(f[q], store_scale<Q, T>(q), J);
            // downstream neighbour x + e_q: the row of the mirrored pull
            if (decltype(sel)::value && R.wall[2 - j][2 - k]) {
                Pair<T>::template st2s<q>(element<kRag, kPlain>(io.out[o], own), v, seed);
            } else {
                const int row = R.off[2 - j][2 - k];
                const auto dst = [&](int x) { return element<kRag, kPlain>(io.out[q], row + x); };
                if constexpr (i == 0)
                    Pair<T>::template st2s<q>(dst(Y.x0), v, seed);
                else if constexpr (i == 1)
                    Pair<T>::template st1x2s<q>(dst(Y.x0 + 1), dst(Y.xp), v, seed);
                else
                    Pair<T>::template st1x2s<q>(dst(Y.xm), dst(Y.x0), v, seed);
            }
        });
    };
    if (edge)
        store(std::integral_constant<bool, kWalls>{});
    else
        store(std::false_type{});
}

// Initial state from FP64 density and velocity fields.
template <int Q, typename T>
__global__ void __launch_bounds__(128) init_kernel(const StepIO<T> io, const StepArgs a,
                                                   const double *__restrict__ rho,
                                                   const double *__restrict__ u) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, x, y, z);
    float Fx, Fy, Fz;
    cell_force(a, c, N, Fx, Fy, Fz);
    float f[Q];
    equilibrium<Q>(float(rho[c] - 1.0), float(u[c]), float(u[N + c]), float(u[2 * N + c]), Fx, Fy,
                   Fz, f);
    scatter_state<Q, T>(io, a.g, x, y, z, f);
}

// Load a dense FP64 state [Q][N] (pre-collision values at their own cells).
template <int Q, typename T>
__global__ void __launch_bounds__(128) set_state_kernel(const StepIO<T> io, const Grid g,
                                                        const double *__restrict__ fin) {
    int x, y, z;
    if (!cell_coords(g, x, y, z)) return;
    const long long N = (long long)g.nx * g.ny * g.nz;
    const double *src = fin + dense_index(g, x, y, z);
    double v[Q];  // all loads before the conversions, whose branches would order them
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = __ldcs(src + q * N);
    float f[Q];
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        f[q] = deviation<Q, q>(v[q]);
    });
    scatter_state<Q, T>(io, g, x, y, z, f);
}

// BF16 momentum references of a state being loaded (reference array 0), one
// thread per pair of cells: J = 3 x the mean velocity of the pair, from the
// velocity field u when given, else from the momentum of the distributions
// f (dense FP64 [Q][N]).  Any J would do as long as the values are stored
// and read against the same one; this one keeps the stored values small.
template <int Q, typename T>
__global__ void __launch_bounds__(128) ref_init_kernel(T *__restrict__ buf, const Grid g,
                                                       const double *__restrict__ u,
                                                       const double *__restrict__ f) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    const int x0 = 2 * t;
    if (x0 >= g.nx || y >= g.ny) return;
    const long long N = (long long)g.nx * g.ny * g.nz;
    const long long c = dense_index(g, x0, y, z);
    const int n = (x0 + 1 < g.nx) ? 2 : 1;
    float v[2][3];
    for (int m = 0; m < n; ++m)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double sum = 0.0;
            if (u) {
                sum = u[d * N + c + m];
            } else {
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int e = d == 0 ? ex<Q>(q) : d == 1 ? ey<Q>(q) : ez<Q>(q);
                    if (e) sum += e * f[q * N + c + m];
                }
            }
            v[m][d] = float(sum);
        }
    float4 J = n == 2 ? make_float4(1.5f * (v[0][0] + v[1][0]), 1.5f * (v[0][1] + v[1][1]),
                                    1.5f * (v[0][2] + v[1][2]), 0.0f)
                      : make_float4(3.0f * v[0][0], 3.0f * v[0][1], 3.0f * v[0][2], 0.0f);
    J.w = J.x;  // stored as (Jx, Jy, Jz, Jx): see load_ref
    ref_array<Q>(buf, g.pop, 0)[((long long)(z * g.ny + y) * g.px + x0) >> 1] = J;
}

// Read the state back as dense FP64 [Q][N].
template <int Q, typename T>
__global__ void __launch_bounds__(128) get_state_kernel(const StepIO<T> io, const Grid g,
                                                        double *__restrict__ fout) {
    int x, y, z;
    if (!cell_coords(g, x, y, z)) return;
    const long long N = (long long)g.nx * g.ny * g.nz;
    double *dst = fout + dense_index(g, x, y, z);
    float f[Q];
    gather<Q, T>(io, g, x, y, z, f);
    static_for<Q>([&](auto iq) {
        constexpr int q = decltype(iq)::value;
        __stcs(dst + q * N, weight_plus<Q, q>(f[q]));
    });
}

template <int Q>
__device__ __forceinline__ void moments(const float (&f)[Q], float &drho, float &jx, float &jy,
                                        float &jz) {
    drho = jx = jy = jz = 0.0f;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        drho += f[a];
        if (ex<Q>(a)) jx += ex<Q>(a) * f[a];
        if (ey<Q>(a)) jy += ey<Q>(a) * f[a];
        if (ez<Q>(a)) jz += ez<Q>(a) * f[a];
    }
}

// Density and velocity (Eqs. densitycalculation, velocitycalculation).
template <int Q, typename T>
__global__ void __launch_bounds__(128) macro_kernel(const StepIO<T> io, const StepArgs a,
                                                    float *__restrict__ rho,
                                                    float *__restrict__ u) {
    int x, y, z;
    if (!cell_coords(a.g, x, y, z)) return;
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    const long long c = dense_index(a.g, x, y, z);
    float f[Q];
    gather<Q, T>(io, a.g, x, y, z, f);
    float drho, jx, jy, jz, Fx, Fy, Fz;
    moments<Q>(f, drho, jx, jy, jz);
    cell_force(a, c, N, Fx, Fy, Fz);
    const float r = 1.0f + drho, ir = 1.0f / r;
    if (rho) rho[c] = r;
    if (u) {
        u[c] = (jx + 0.5f * Fx) * ir;
        u[N + c] = (jy + 0.5f * Fy) * ir;
        u[2 * N + c] = (jz + 0.5f * Fz) * ir;
    }
}

// Global sums.  Blocks of at most 128 threads, shaped like the other per-cell
// kernels' (short rows share a block), stride over the rows of the grid, at
// most eight blocks per SM resident; each leaves one partial record of 4
// doubles, added up in a fixed order by reduce_final_kernel.  A cell's moments
// are FP32 sums of its stored deviations; the running sums across cells are
// FP64.
constexpr int kFinalThreads = 256;
constexpr int kRedBlocks = kSMs * 8;

struct RedLaunch {
    dim3 block;
    int blocks;
};
inline RedLaunch red_launch(const Grid &g) {
    RedLaunch L;
    L.block = cell_launch(g).block;
    const long long groups = ((long long)g.ny * g.nz + L.block.y - 1) / L.block.y;
    L.blocks = int(groups < kRedBlocks ? groups : kRedBlocks);
    return L;
}

// fn(x, y, z, dense cell index) over the block's share of the cells.
template <typename Fn>
__device__ __forceinline__ void for_cells(const Grid &g, Fn &&fn) {
    const unsigned rows = unsigned(g.ny) * unsigned(g.nz);  // ny, nz <= 65535
    for (unsigned row = blockIdx.x * blockDim.y + threadIdx.y; row < rows;
         row += gridDim.x * blockDim.y) {
        const int z = int(row / unsigned(g.ny)), y = int(row - unsigned(z) * unsigned(g.ny));
        for (int x = threadIdx.x; x < g.nx; x += blockDim.x)
            fn(x, y, z, (long long)row * g.nx + x);
    }
}

// Sum of the threads' acc[K] over the block (whole warps, at most four), in a
// fixed order; valid in thread 0.
template <int K>
__device__ __forceinline__ void block_sum(double (&acc)[K]) {
    __shared__ double sh[K][4];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const int warps = int(blockDim.x * blockDim.y) >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], d);
        if ((t & 31) == 0) sh[k][t >> 5] = acc[k];
    }
    __syncthreads();
    if (t == 0)
#pragma unroll
        for (int k = 0; k < K; ++k)
            for (int w = 1; w < warps; ++w) acc[k] += sh[k][w];
}

// Partial sums of (rho - 1, rho u).
template <int Q, typename T>
__global__ void __launch_bounds__(128, 8) conservation_kernel(const StepIO<T> io, const StepArgs a,
                                                              double *__restrict__ part) {
    const long long N = (long long)a.g.nx * a.g.ny * a.g.nz;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for_cells(a.g, [&](int x, int y, int z, long long c) {
        float f[Q];
        gather<Q, T>(io, a.g, x, y, z, f);
        float drho, jx, jy, jz, Fx, Fy, Fz;
        moments<Q>(f, drho, jx, jy, jz);
        cell_force(a, c, N, Fx, Fy, Fz);
        acc[0] += widen(drho);
        acc[1] += widen(jx + 0.5f * Fx);
        acc[2] += widen(jy + 0.5f * Fy);
        acc[3] += widen(jz + 0.5f * Fz);
    });
    block_sum(acc);
    if (threadIdx.x == 0 && threadIdx.y == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) part[4 * blockIdx.x + k] = acc[k];
}

// Launchers.  kernels.cu holds their explicit instantiations; api.cu sees them
// through extern declarations (the macros below).
inline unsigned long long splat_bits(float v) {
    unsigned int u;
    memcpy(&u, &v, 4);
    return (unsigned long long)u << 32 | u;
}

// weighted: for collide27_g on weight-scaled inputs, (1 - omega) / 216.
inline PackedRates packed_rates(const StepArgs &a, bool weighted = false) {
    PackedRates p;
    for (int b = 0; b < 15; ++b) p.w15[b] = splat_bits(a.w[b] * k15_inv(b));
    for (int b = 0; b < 27; ++b) {
        const float w = a.w[b], nw = -a.w[b];
        const float omw = weighted ? (1.0f - a.w[b]) / 216.0f : 1.0f - a.w[b];
        unsigned int uw, unw, uomw;
        memcpy(&uw, &w, 4);
        memcpy(&unw, &nw, 4);
        memcpy(&uomw, &omw, 4);
        p.w[b] = (unsigned long long)uw << 32 | uw;
        p.nw[b] = (unsigned long long)unw << 32 | unw;
        p.omw[b] = (unsigned long long)uomw << 32 | uomw;
    }
    return p;
}

// D3Q27: the rates from the trace on (omega_9 .. omega_26) are all exactly
// 1, the paper's choice for every non-shear moment, so the pair kernels can
// take the kEq form of the relaxation (relax27: the same arithmetic, with
// the work that only fed those moments dropped).
inline bool higher_rates_are_one(const StepArgs &a) {
    for (int b = 9; b < 27; ++b)
        if (a.w[b] != 1.0f) return false;
    return true;
}

// Plane pointers of an input and an output state buffer (either may be null:
// not accessed by the kernel then) and their BF16 reference arrays.
template <int Q, typename T>
StepIO<T> step_io(const void *fin, void *fout, const Grid &g, int ref_in = 0, int ref_out = 0) {
    StepIO<T> io{};
    for (int q = 0; q < Q; ++q) {
        if (fin) io.in[q] = static_cast<const T *>(fin) + q * g.pop;
        if (fout) io.out[q] = static_cast<T *>(fout) + q * g.pop;
    }
    if (Storage<T>::kRef && fin)
        io.ref_in = ref_array<Q>(static_cast<const T *>(fin), g.pop, ref_in);
    if (Storage<T>::kRef && fout) io.ref_out = ref_array<Q>(static_cast<T *>(fout), g.pop, ref_out);
    return io;
}
// The same for a kernel that only reads the state, in whichever layout.
template <int Q, typename T>
StepIO<T> read_io(const void *f, const Grid &g) {
    return step_io<Q, T>(f, nullptr, g, g.layout == kAASwapped ? 1 : 0);
}

// Launch geometry of the kernels with two cells per thread over `row` cells per
// row (stored_row: to the end of the last sector).
inline CellLaunch pair_launch(const Grid &g, int row) {
    Grid half = g;
    half.nx = (row + 1) / 2;
    return cell_launch(half);
}

// Whether a grid takes the instantiations for ragged rows (kRag): rows that do
// not fill their last sector, or planes beyond 32-bit byte offsets (element()).
template <typename T>
bool ragged(const Grid &g) {
    return stored_row<T>(g.nx) != g.nx || g.pop * (long long)sizeof(T) > (1ll << 32);
}

// Grids of odd rows take the one-cell step kernel where its launch leaves no SM
// more than this many warps: a step is one thread's chain of instructions there.
// us a step, one cell / two cells per thread, FP32, warps in brackets: D3Q27
// periodic 23^3 (4) 2.25 / 2.57, 257 x 10 x 9 (6) 2.44 / 2.82, 25^3 (8) 2.72 / 2.63;
// walled 23^3 2.31 / 3.21, 27^3 (8) 2.82 / 3.29, 33^3 (16) 3.79 / 3.27; D3Q15
// periodic with force 23^3 1.87 / 2.31, walled 23^3 2.06 / 2.25, 27^3 2.36 / 2.32,
// without force 2.06 / 2.12.  Rows of one cell take the two-cell kernel (1 x 100 x
// 100 walled 6.94 / 5.39).
// 16-bit storage (17^3): between walls, where the two-cell kernel's wall selects cost
// most (D3Q27 BF16 2.8 / 5.6, at 33^3 4.8 / 5.8, FP16 2.70 / 3.53; D3Q15 BF16 2.25 /
// 2.94, FP16 2.18 / 2.44), and D3Q27 periodic (BF16 2.31 / 3.27, FP16 at general rates
// 2.25 / 2.70, at the rate-1 form 2.3 / 2.4 but 0.9x at 3 x 43 x 43).
template <int Q, typename T, bool kWalls, bool kForm>
constexpr int kOneCellWarps =
    std::is_same<T, float>::value ? (kWalls || Q == 15 ? 8 : 6)
    : Storage<T>::kRef            ? (kWalls ? (Q == 27 ? 16 : 12) : (Q == 27 ? 6 : 0))
    : kWalls                      ? (Q == 27 ? 12 : 6)
                                  : (Q == 27 && !kForm ? 6 : 0);

// kForm: the rate-1 relaxation (D3Q27), a force anywhere (D3Q15).
template <int Q, typename T, bool kWalls, bool kForm>
void launch_step_kernel(const StepIO<T> &io, const StepArgs &a, const PackedRates &pr,
                      cudaStream_t st) {
    if constexpr (kOneCellWarps<Q, T, kWalls, kForm> > 0) {
        const CellLaunch L = cell_launch(a.g);
        if (a.g.nx % 2 && a.g.nx > 1 && L.sm_warps() <= kOneCellWarps<Q, T, kWalls, kForm>) {
            step1_kernel<Q, T, kWalls, kForm><<<L.grid, L.block, 0, st>>>(io, a);
            return;
        }
    }
    const CellLaunch L = pair_launch(a.g, stored_row<T>(a.g.nx));
    // grids of short rows are small, and a second copy of the loads (pull_pairs)
    // costs them more than it saves: D3Q27 FP32 between walls, 16^3 3.55 / 3.05
    // us, 16 x 64 x 64 4.13 / 3.75 us with / without it
    const bool is_short = L.block.x < 32 && (Storage<T>::kRef || !ragged<T>(a.g));
    if constexpr (Storage<T>::kRef && kWalls) {
        // BF16 in ragged rows too (24^3: D3Q27 5.1 / 5.7, D3Q15 2.76 / 2.89; FP32 and FP16
        // up to 7 % slower)
        if (is_short && ragged<T>(a.g)) {
            if constexpr (Q == 27)
                step2_kernel<T, true, kForm, true, true><<<L.grid, L.block, 0, st>>>(io, a, pr);
            else
                step2_q15_kernel<T, true, kForm, true, true>
                    <<<L.grid, L.block, 0, st>>>(io, a, pr);
            return;
        }
    }
    if constexpr (Q == 27) {
        if constexpr (kWalls) {
            if (is_short) {
                step2_kernel<T, true, kForm, false, true><<<L.grid, L.block, 0, st>>>(io, a, pr);
                return;
            }
        }
        if (ragged<T>(a.g))
            step2_kernel<T, kWalls, kForm, true><<<L.grid, L.block, 0, st>>>(io, a, pr);
        else
            step2_kernel<T, kWalls, kForm, false><<<L.grid, L.block, 0, st>>>(io, a, pr);
    } else {
        // (FP32 and FP16 the other way round: 16^3 2.27 / 2.47, 16 x 64 x 64 2.91 /
        // 3.01 us with / without it; BF16 2.78 / 2.72)
        if constexpr (kWalls && Storage<T>::kRef) {
            if (is_short) {
                step2_q15_kernel<T, true, kForm, false, true>
                    <<<L.grid, L.block, 0, st>>>(io, a, pr);
                return;
            }
        }
        if (ragged<T>(a.g))
            step2_q15_kernel<T, kWalls, kForm, true><<<L.grid, L.block, 0, st>>>(io, a, pr);
        else
            step2_q15_kernel<T, kWalls, kForm, false><<<L.grid, L.block, 0, st>>>(io, a, pr);
    }
}

// Ragged rows (kRag) take their own instantiation of the two-cell kernels, so
// that the others keep immediate offsets.
template <int Q, typename T>
cudaError_t launch_step(const void *fin, void *fout, const StepArgs &a, cudaStream_t st) {
    const StepIO<T> io = step_io<Q, T>(fin, fout, a.g);
    const bool walls = a.g.bc != 0;
    if constexpr (std::is_same<T, float>::value) {
        if (a.sr32) {
            const CellLaunch L = cell_launch(a.g);
            if (walls)
                step_sr32_kernel<Q, true><<<L.grid, L.block, 0, st>>>(io, a);
            else
                step_sr32_kernel<Q, false><<<L.grid, L.block, 0, st>>>(io, a);
            return cudaGetLastError();
        }
    }
    const PackedRates pr = packed_rates(a, kFoldedLoad<Q, T>());
    const bool form = Q == 27 ? higher_rates_are_one(a) : a.has_force != 0;
    if (walls && form)
        launch_step_kernel<Q, T, true, true>(io, a, pr, st);
    else if (walls)
        launch_step_kernel<Q, T, true, false>(io, a, pr, st);
    else if (form)
        launch_step_kernel<Q, T, false, true>(io, a, pr, st);
    else
        launch_step_kernel<Q, T, false, false>(io, a, pr, st);
    return cudaGetLastError();
}

template <int Q, typename T, bool kEq, bool kForce, bool kRag>
void launch_aa_kernels(const StepIO<T> &io, const StepArgs &a, const PackedRates &pr, bool even,
                       const CellLaunch &L, cudaStream_t st) {
    if (even && a.g.bc)
        aa_even_kernel<Q, T, true, kEq, kForce, kRag><<<L.grid, L.block, 0, st>>>(io, a, pr);
    else if (even)
        aa_even_kernel<Q, T, false, kEq, kForce, kRag><<<L.grid, L.block, 0, st>>>(io, a, pr);
    else if (a.g.bc)
        aa_odd_kernel<Q, T, true, kEq, kForce, kRag><<<L.grid, L.block, 0, st>>>(io, a, pr);
    else
        aa_odd_kernel<Q, T, false, kEq, kForce, kRag><<<L.grid, L.block, 0, st>>>(io, a, pr);
}

// One in-place (AA) step on buffer buf: even (kAANatural -> kAASwapped) or
// odd (kAASwapped -> kAANatural).  nx must be even.  D3Q27 takes the rate-1
// form when omega_9..26 are all 1; D3Q15 the force-free cascade when there is
// no force.
template <int Q, typename T>
cudaError_t launch_step_aa(void *buf, const StepArgs &a, bool even, cudaStream_t st) {
    // BF16 references: array 0 for the natural layout, 1 for the swapped one
    const StepIO<T> io = step_io<Q, T>(buf, buf, a.g, even ? 0 : 1, even ? 1 : 0);
    const CellLaunch L = pair_launch(a.g, stored_row<T>(a.g.nx));
    const PackedRates pr = packed_rates(a, kFoldedLoad<Q, T>());
    const auto launch = [&](auto form) {
        constexpr bool kEq = Q == 27 && decltype(form)::value;
        constexpr bool kForce = Q == 27 || decltype(form)::value;
        if (ragged<T>(a.g))
            launch_aa_kernels<Q, T, kEq, kForce, true>(io, a, pr, even, L, st);
        else
            launch_aa_kernels<Q, T, kEq, kForce, false>(io, a, pr, even, L, st);
    };
    if (Q == 27 ? higher_rates_are_one(a) : a.has_force != 0)
        launch(std::true_type{});
    else
        launch(std::false_type{});
    return cudaGetLastError();
}

// BF16: the references of the state being loaded, before its values.
template <int Q, typename T>
cudaError_t launch_ref_init(T *buf, const Grid &g, const double *u, const double *f,
                            cudaStream_t st) {
    const CellLaunch L = pair_launch(g, g.nx);
    ref_init_kernel<Q, T><<<L.grid, L.block, 0, st>>>(buf, g, u, f);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_init(void *buf, const StepArgs &a, const double *rho, const double *u,
                        cudaStream_t st) {
    if constexpr (Storage<T>::kRef) {
        const cudaError_t e = launch_ref_init<Q, T>(static_cast<T *>(buf), a.g, u, nullptr, st);
        if (e != cudaSuccess) return e;
    }
    const CellLaunch L = cell_launch(a.g);
    init_kernel<Q, T><<<L.grid, L.block, 0, st>>>(step_io<Q, T>(nullptr, buf, a.g), a, rho, u);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_set_state(void *buf, const Grid &g, const double *f, cudaStream_t st) {
    if constexpr (Storage<T>::kRef) {
        const cudaError_t e = launch_ref_init<Q, T>(static_cast<T *>(buf), g, nullptr, f, st);
        if (e != cudaSuccess) return e;
    }
    const CellLaunch L = cell_launch(g);
    set_state_kernel<Q, T><<<L.grid, L.block, 0, st>>>(step_io<Q, T>(nullptr, buf, g), g, f);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_get_state(const void *buf, const Grid &g, double *f, cudaStream_t st) {
    const CellLaunch L = cell_launch(g);
    get_state_kernel<Q, T><<<L.grid, L.block, 0, st>>>(read_io<Q, T>(buf, g), g, f);
    return cudaGetLastError();
}

template <int Q, typename T>
cudaError_t launch_macro(const void *buf, const StepArgs &a, float *rho, float *u,
                         cudaStream_t st) {
    const CellLaunch L = cell_launch(a.g);
    macro_kernel<Q, T><<<L.grid, L.block, 0, st>>>(read_io<Q, T>(buf, a.g), a, rho, u);
    return cudaGetLastError();
}

// Partial records of the conservation sums: red_launch(g).blocks of them.
template <int Q, typename T>
cudaError_t launch_conservation(const void *buf, const StepArgs &a, double *part,
                                cudaStream_t st) {
    const RedLaunch L = red_launch(a.g);
    conservation_kernel<Q, T><<<L.blocks, L.block, 0, st>>>(read_io<Q, T>(buf, a.g), a, part);
    return cudaGetLastError();
}

// Final reduction of the per-block partials to 4 doubles (one block).
cudaError_t launch_reduce_final(const double *part, int blocks, double *out, cudaStream_t st);

#define LBM_INSTANTIATE_STEP(EXT, Q, T) \
    EXT template cudaError_t launch_step<Q, T>(const void *, void *, const StepArgs &, cudaStream_t);

#define LBM_INSTANTIATE_INPLACE(EXT, Q, T) \
    EXT template cudaError_t launch_step_aa<Q, T>(void *, const StepArgs &, bool, cudaStream_t);

#define LBM_INSTANTIATE_STATE(EXT, Q, T)                                                         \
    EXT template cudaError_t launch_init<Q, T>(void *, const StepArgs &, const double *,         \
                                               const double *, cudaStream_t);                  \
    EXT template cudaError_t launch_set_state<Q, T>(void *, const Grid &, const double *,        \
                                                    cudaStream_t);                             \
    EXT template cudaError_t launch_get_state<Q, T>(const void *, const Grid &, double *,        \
                                                    cudaStream_t);                             \
    EXT template cudaError_t launch_macro<Q, T>(const void *, const StepArgs &, float *, float *, \
                                                cudaStream_t);                                 \
    EXT template cudaError_t launch_conservation<Q, T>(const void *, const StepArgs &, double *, \
                                                       cudaStream_t);

}  // namespace lbm
