// Far-field vector amplitudes of the dipole array ("Averaging over Scattering
// Directions", "Scattering by Finite Targets: The Mueller Matrix"):
//
//   F_r(n_d) = k^2 (I - n_d n_d) sum_j P_{r,j} exp(-i k n_d . r_j)
//
// for every right-hand side r and scattering direction n_d (the scattered
// field is exp(ikR)/R F at distance R along n_d, so dC_sca/dOmega = |F|^2).
// The sites lie on a lattice, so the phase factors separate,
// exp(-ik n.r) = ex(ix) ey(iy) ez(iz), with one table per axis and direction
// (FP64 sincos, rounded to the arithmetic type).
#include <cuda_runtime.h>

#include <algorithm>

#include "farfield.h"
#include "krylov_dev.cuh"
#include "profiler.h"

namespace dda {

namespace {

constexpr int kFFWarps = 8;
// Rows a block sums before its totals go to FP64: a bound on the length of the
// sums in the arithmetic type.
constexpr int kFFRows = 256;
constexpr int kFFMaxSmem = 227 * 1024;  // dynamic shared memory a block can have

// n consecutive complex numbers from shared memory, in 16-byte words where they fit
template <int n, typename C> __device__ __forceinline__ void read_words(C (&v)[n], const C* s) {
    if constexpr (sizeof(C) == 8 && n % 2 == 0) {
#pragma unroll
        for (int i = 0; i < n; i += 2) {
            const float4 q = *reinterpret_cast<const float4*>(s + i);
            v[i] = make_float2(q.x, q.y);
            v[i + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < n; ++i) v[i] = s[i];
    }
}

// The sum over a lattice row x of P ex needs one complex product per site and
// component; ey ez multiplies once per row.  (Forming the whole phase at
// every site took 8 of its 20 multiply-adds.)  A lane holds TD directions and
// runs over the sites, which its warp stages 32 at a time in shared memory
// and reads back by broadcast; ex comes from the block's table [nx][32 TD],
// whose words the lanes of a warp read consecutively and the block's eight
// warps, on rows of their own, share.  Both polarizations of a direction (NR
// = 2) share it too: per site and lane 12 TD NR multiply-adds for TD table
// words.  Bound by the FP32 pipes; 16 RHS x 2172 directions x 102984 sites:
// 5.60 -> 2.30 ms with two directions a lane, 2.1 ms with four (at two thirds of
// the issue slots: multiply-adds of three different registers run at 87 of 128
// lanes).  In packed pairs, which need P's parts twice in shared memory, it took
// 2.6 ms.
template <typename C, int NR, int TD>
__global__ void __launch_bounds__(kFFWarps * 32, 2)
    k_farfield(const double2* __restrict__ P, int64_t N, const int* __restrict__ rows,
               const int* __restrict__ row_start, int nrows, int per_chunk, const int* __restrict__ lat_of, int nxe,
               int nye, FarGeom f, const C* __restrict__ tabs, const double* __restrict__ dirs, double kd,
               double2* __restrict__ F) {
    constexpr int ND = 32 * TD, NC = NR * 3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tab = reinterpret_cast<C*>(smem_raw);  // [nx][ND]
    C* buf = tab + f.nx * ND;                 // [warps][32][NC]
    int* bix = reinterpret_cast<int*>(buf + kFFWarps * 32 * NC);
    const int grp = blockIdx.y, d0 = blockIdx.x * ND, Lt = f.nx + f.ny + f.nz;
    const C* gt = tabs + (int64_t)grp * Lt * f.ndp + d0;
    for (int e = threadIdx.x; e < f.nx * ND; e += kFFWarps * 32) tab[e] = gt[(int64_t)(e / ND) * f.ndp + e % ND];
    __syncthreads();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    C* wb = buf + warp * 32 * NC;
    int* wi = bix + warp * 32;
    // direction t of a lane: neighbouring pairs, one 16-byte word apart from the
    // next lane's, the second pair of four 64 directions on
    auto dir = [&](int t) { return TD == 4 ? t / 2 * 64 + lane * 2 + t % 2 : lane * TD + t; };
    const C* tl = tab + dir(0);
    const double2* Pg = P + (int64_t)grp * NC * N;
    C tot[TD][NC];
#pragma unroll
    for (int t = 0; t < TD; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) tot[t][c] = czero<C>();
    const int row1 = min(nrows, ((int)blockIdx.z + 1) * per_chunk);
    for (int row = blockIdx.z * per_chunk + warp; row < row1; row += kFFWarps) {
        const int id = rows[row], iy = id % nye, iz = id / nye, s1 = row_start[row + 1];
        C acc[TD][NC];
#pragma unroll
        for (int t = 0; t < TD; ++t)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[t][c] = czero<C>();
        for (int s = row_start[row]; s < s1; s += 32) {
            const int m = min(32, s1 - s);
            __syncwarp();
            if (lane < m) {
                wi[lane] = (lat_of[s + lane] - id * nxe) * ND;
#pragma unroll
                for (int c = 0; c < NC; ++c) wb[lane * NC + c] = ccast<C>(Pg[c * N + s + lane]);
            }
            __syncwarp();
#pragma unroll 4
            for (int i = 0; i < m; ++i) {
                const C* ex = tl + wi[i];
                C e[TD], p[NC];
                if constexpr (TD == 4) {
                    read_words(reinterpret_cast<C(&)[2]>(e[0]), ex);
                    read_words(reinterpret_cast<C(&)[2]>(e[2]), ex + 64);
                } else {
                    read_words(e, ex);
                }
                read_words(p, wb + i * NC);
#pragma unroll
                for (int t = 0; t < TD; ++t)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        acc[t][c].x += p[c].x * e[t].x;
                        acc[t][c].y += p[c].x * e[t].y;
                        acc[t][c].x -= p[c].y * e[t].y;
                        acc[t][c].y += p[c].y * e[t].x;
                    }
            }
        }
#pragma unroll
        for (int t = 0; t < TD; ++t) {
            const int d = dir(t);
            const C ph = cmul(gt[(int64_t)(f.nx + iy) * f.ndp + d], gt[(int64_t)(f.nx + f.ny + iz) * f.ndp + d]);
#pragma unroll
            for (int c = 0; c < NC; ++c) tot[t][c] = cadd(tot[t][c], cmul(acc[t][c], ph));
        }
    }
    __syncthreads();
    C* red = reinterpret_cast<C*>(smem_raw);  // [warps][NC][ND]
#pragma unroll
    for (int t = 0; t < TD; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) red[(warp * NC + c) * ND + dir(t)] = tot[t][c];
    __syncthreads();
    for (int e = threadIdx.x; e < ND * NR; e += kFFWarps * 32) {
        const int r = e / ND, td = e % ND, d = d0 + td;
        if (d >= f.ndir) continue;
        double2 s[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s[a] = make_double2(0.0, 0.0);
            for (int w = 0; w < kFFWarps; ++w) {
                const C v = red[(w * NC + r * 3 + a) * ND + td];
                s[a].x += (double)v.x;
                s[a].y += (double)v.y;
            }
        }
        // (I - n n) s, times k^2; partial sums of the row chunks add atomically
        const double* n = dirs + ((int64_t)grp * f.ndir + d) * 3;
        const double2 ns = make_double2(n[0] * s[0].x + n[1] * s[1].x + n[2] * s[2].x,
                                        n[0] * s[0].y + n[1] * s[1].y + n[2] * s[2].y);
        double2* out = F + ((int64_t)(grp * NR + r) * f.ndir + d) * 3;
        const double k2 = kd * kd;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            atomicAdd(&out[a].x, k2 * (s[a].x - n[a] * ns.x));
            atomicAdd(&out[a].y, k2 * (s[a].y - n[a] * ns.y));
        }
    }
}

// The tables of launch_phase_tables.  An axis is symmetric about its centre, so
// one FP64 sincos serves the indices i and n - 1 - i (and a group of RHS one
// table: 556 -> 99 us for 16 RHS x 2172 directions of a 96x64x32 lattice).
template <typename C>
__global__ void k_phase_tables(FarGeom f, int groups, double kd, const double* __restrict__ dirs,
                               C* __restrict__ tabs) {
    const int hx = (f.nx + 1) / 2, hy = (f.ny + 1) / 2, hz = (f.nz + 1) / 2, per = hx + hy + hz;
    const int Lt = f.nx + f.ny + f.nz;
    const int64_t total = (int64_t)groups * per * f.ndp;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int d = (int)(e % f.ndp), h = (int)((e / f.ndp) % per), grp = (int)(e / ((int64_t)f.ndp * per));
        const int a = h < hx ? 0 : (h < hx + hy ? 1 : 2);
        const int i = a == 0 ? h : (a == 1 ? h - hx : h - hx - hy), n = a == 0 ? f.nx : (a == 1 ? f.ny : f.nz);
        const int at = a == 0 ? 0 : (a == 1 ? f.nx : f.nx + f.ny);
        double2 v = make_double2(0.0, 0.0);
        if (d < f.ndir) sincos(-kd * dirs[((int64_t)grp * f.ndir + d) * 3 + a] * (i - 0.5 * (n - 1)), &v.y, &v.x);
        C* out = tabs + ((int64_t)grp * Lt + at) * f.ndp + d;
        out[(int64_t)(n - 1 - i) * f.ndp] = ccast<C>(make_double2(v.x, -v.y));
        out[(int64_t)i * f.ndp] = ccast<C>(v);
    }
}

}  // namespace

template <typename C>
cudaError_t launch_phase_tables(const FarGeom& f, int groups, double kd, const double* dirs, C* tabs,
                                cudaStream_t st) {
    const int64_t total = (int64_t)groups * ((f.nx + 1) / 2 + (f.ny + 1) / 2 + (f.nz + 1) / 2) * f.ndp;
    const int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
    PROF_BEGIN(st);
    k_phase_tables<C><<<blocks, 256, 0, st>>>(f, groups, kd, dirs, tabs);
    PROF_END(KK_FARFIELD, 1, st);
    return cudaGetLastError();
}
template cudaError_t launch_phase_tables<float2>(const FarGeom&, int, double, const double*, float2*, cudaStream_t);
template cudaError_t launch_phase_tables<double2>(const FarGeom&, int, double, const double*, double2*, cudaStream_t);

template <typename C>
cudaError_t launch_farfield(const Geom& g, const DevTarget& tg, const FarGeom& f, int groups, int NR, const double2* P,
                            const C* tabs, const double* dirs, double kd, double2* F, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(F, 0, (size_t)groups * NR * f.ndir * 3 * sizeof(double2), st);
    if (e != cudaSuccess) return e;
    // directions per lane: four while two blocks' tables fit an SM, else two; one
    // in FP64 (whose table words are twice as wide)
    constexpr int TW = sizeof(C) == 8 ? 4 : 1, TN = sizeof(C) == 8 ? 2 : 1;
    auto smem = [&](int td) {
        const size_t work =
            (size_t)f.nx * 32 * td * sizeof(C) + (size_t)kFFWarps * 32 * (NR * 3 * sizeof(C) + sizeof(int));
        return std::max(work, (size_t)kFFWarps * NR * 3 * 32 * td * sizeof(C));
    };
    const bool wide = TW > TN && smem(TW) <= 112 * 1024;
    const int ND = 32 * (wide ? TW : TN);
    const size_t sm = smem(wide ? TW : TN);
    // row chunks: at most kFFRows rows, and enough blocks for two waves of the 152 SMs
    const int tiles = (f.ndir + ND - 1) / ND;
    const int64_t want = (4 * 152 + (int64_t)tiles * groups - 1) / ((int64_t)tiles * groups);
    const int chunks = (int)std::min<int64_t>(
        65535, std::max<int64_t>((tg.nrows + kFFRows - 1) / kFFRows,
                                 std::min<int64_t>(want, (tg.nrows + kFFWarps - 1) / kFFWarps)));
    const int per_chunk = (tg.nrows + chunks - 1) / chunks;
    auto go = [&](auto kern) -> cudaError_t {
        // the limit, not sm: another thread's context may set it between here and the launch
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kFFMaxSmem);
        if (e != cudaSuccess) return e;
        PROF_BEGIN(st);
        kern<<<dim3(tiles, groups, chunks), kFFWarps * 32, sm, st>>>(P, g.N, tg.rows, tg.row_start, tg.nrows, per_chunk,
                                                                    tg.lat_of, g.nx, g.ny, f, tabs, dirs, kd, F);
        PROF_END(KK_FARFIELD, groups * NR, st);
        return cudaGetLastError();
    };
    if (wide) return NR == 2 ? go(k_farfield<C, 2, TW>) : go(k_farfield<C, 1, TW>);
    return NR == 2 ? go(k_farfield<C, 2, TN>) : go(k_farfield<C, 1, TN>);
}

template cudaError_t launch_farfield<float2>(const Geom&, const DevTarget&, const FarGeom&, int, int, const double2*,
                                             const float2*, const double*, double, double2*, cudaStream_t);
template cudaError_t launch_farfield<double2>(const Geom&, const DevTarget&, const FarGeom&, int, int, const double2*,
                                              const double2*, const double*, double, double2*, cudaStream_t);

}  // namespace dda
