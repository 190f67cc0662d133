// The y and z transforms of the complex64 matvec in one pass over slabs.
//
// After the x-forward pass every kx is independent of every other: at fixed
// (RHS, kx) the rest of the convolution -- FFT along y, FFT along z, the 3x3
// product with the Green tensor, both inverses -- maps one slab of
// 3 nz ny numbers to one of the same size.  k_slab keeps the slab in shared
// memory from end to end, so the matvec moves 24 numbers per lattice site and
// RHS between its passes instead of 72 (the separate passes write the
// y-transformed half-spectrum, twice the size, and carry it through the z
// pass).  The buffer between the passes is kx-major,
//     U [R][3][Lx][nz ny],
// one contiguous block per slab and component; the x passes stage 16 rows in
// shared memory anyway and write or read it 16 rows at a time.
//
// Phases of a block (one slab), in place on S [3][nz][RS] (RS >= Ly):
//   A  rows (c, iz): FFT along y of the ny loaded numbers -> Ly spectrum
//   B  columns (ky): all three components, FFT along z (input half zero),
//      product, inverse FFT, lattice half kept
//   C  rows: inverse FFT along y, lattice half stored
// The arithmetic is packed (pair.cuh): A and C run rows iz and iz + nz/2 in the
// two halves, B the columns ky and Ly-ky.  These two share their Green tensor:
// its entries xy and yz change sign under ky -> -ky and the others do not, so
// with the y component of the mirrored column negated on the way in and out
// both halves multiply by the same six numbers.  (ky = 0 and Ly/2 are their own
// mirrors and form a pair with a tensor each; there xy and yz vanish.)
// Likewise the sign of kx > Lx/2 (xy and xz) goes into the x component, at A's
// loads and C's stores.
// A pencil lies in NT lanes of one warp, so its exchanges wait for no other
// warp; they use the pencil's own words of S.
// Measured, y + z + y passes before -> this kernel: 96x64x32 ellipsoid, 32 RHS
// 710 -> 470 us; 64^3 sphere, 2 RHS 83 -> 57 us; 48^3, 4 RHS 107 -> 75 us.  Bound by
// latency and dependent issue at 12 warps per SM (issue 49 %, FP32 pipes 52 %,
// shared pipe 70 %): 96 registers hold a thread's points, so 168 x 384 threads
// fill the register file; 512 threads of 128 registers spilled and took 3 % more.
// Whole rounds cost besides: phase B deals 16 column groups to 6 warps (Ly 128, Lz
// 64) or 32 to 12 (128, 128), which fills 89 % of three rounds, and 12 to 8 (96, 96)
// or 6 to 4 (96, 48), 75 % of two; and a launch's slabs come in waves of the SMs.
#pragma once

#include "matvec_impl.cuh"
#include "pair.cuh"

namespace dda {

// Row plans (phases A, C: one component per thread) and column plans (phase
// B: three components in lockstep, 12 registers per point).
template <int L> struct RowPlan;
template <> struct RowPlan<16> : PlanDef<16, 4, 4, 4> {};
template <> struct RowPlan<32> : PlanDef<32, 4, 4, 8> {};
template <> struct RowPlan<48> : PlanDef<48, 4, 4, 4, 3> {};
template <> struct RowPlan<64> : PlanDef<64, 8, 8, 8> {};
template <> struct RowPlan<96> : PlanDef<96, 8, 4, 4, 6> {};
template <> struct RowPlan<128> : PlanDef<128, 8, 8, 16> {};
template <int L> struct ColPlan : RowPlan<L> {};
// 128 points of three components do not fit a thread's registers in a plan
// with one exchange (8 x 16: 192 registers), so the transform is split by
// parity: with only n = 64 inputs x_j, the even frequencies are the n-point
// DFT of x_j and the odd ones that of x_j exp(-i pi j / n), both 8 x 8.  Half
// of a pair's lanes take each, and the inverse's two halves are added across
// lanes at the end.
template <> struct ColPlan<128> : PlanDef<64, 8, 8, 8> {};
template <int LZ> __host__ __device__ constexpr bool col_split() { return ColPlan<LZ>::L != LZ; }
template <int LZ> __host__ __device__ constexpr int col_lanes() { return ColPlan<LZ>::NT * (col_split<LZ>() ? 2 : 1); }

// Column pairs of a warp in phase B, and the row stride of S (8-byte words):
// rows a column steps through shift by the width of the pair group, so that
// the lanes of a half-warp fall on different banks.
template <int LZ> __host__ __device__ constexpr int slab_wt() { return 32 / col_lanes<LZ>(); }
// (adjacent lanes take slab_w adjacent pairs; of eight, the half-warps take four each)
template <int LZ> __host__ __device__ constexpr int slab_w() { return slab_wt<LZ>() < 4 ? slab_wt<LZ>() : 4; }
template <int LZ> __host__ __device__ constexpr int col_pair(int lane) {
    return lane % slab_w<LZ>() + (slab_wt<LZ>() > 4 ? 4 * (lane / 16) : 0);
}
template <int LZ> __host__ __device__ constexpr int col_lane(int lane) {  // place in the pair: u + NT par
    return (lane / slab_w<LZ>()) % col_lanes<LZ>();
}
template <int LY, int LZ> __host__ __device__ constexpr int slab_rs() { return LY + slab_w<LZ>(); }
template <int LY, int LZ> __host__ __device__ constexpr size_t slab_smem() {
    return (size_t)3 * (LZ / 2) * slab_rs<LY, LZ>() * 8 + (size_t)(LY + LZ) * 16;
}
// Threads per SM: 384 of 168 registers, or 256 of 255 where a thread holds 12
// points of the three components.  Blocks per SM by shared memory.
template <int LZ> __host__ __device__ constexpr int slab_sm_threads() { return ColPlan<LZ>::E > 8 ? 256 : 384; }
template <int LY, int LZ> __host__ __device__ constexpr int slab_blocks() {
    const size_t sm = slab_smem<LY, LZ>() + 1024;
    return sm * 3 <= 227 * 1024 && slab_sm_threads<LZ>() == 384 ? 3 : (sm * 2 <= 227 * 1024 ? 2 : 1);
}
// (NB blocks per SM: that, or one block with all the threads where a launch has
// no more slabs than SMs)
template <int LY, int LZ, int NB> __host__ __device__ constexpr int slab_threads() { return slab_sm_threads<LZ>() / NB; }

// A row pencil holds rows q and q + NZ/2, real parts of its exchanges in the one
// and imaginary parts in the other.  The 16 / NT pencils of a half-warp must lie
// NT banks apart; rows lie slab_w apart, so they take every (NT / slab_w)-th row.
template <int LY, int LZ> __host__ __device__ constexpr int slab_row_step() { return RowPlan<LY>::NT / slab_w<LZ>(); }
template <int LY, int LZ> __host__ __device__ constexpr int slab_row(int rp) {
    constexpr int H = 16 / RowPlan<LY>::NT, D = slab_row_step<LY, LZ>();
    static_assert(D >= 1 && (LZ / 4) % (H * D) == 0, "whole groups of rows");
    return rp / (H * D) * (H * D) + rp % H * D + rp / H % D;
}

template <int LY, int LZ> struct RowMapY {
    __host__ __device__ static constexpr LaneMap map() {
        return LaneMap{1, RowPlan<LY>::NT, 32 / RowPlan<LY>::NT, 1, slab_row_step<LY, LZ>() * slab_rs<LY, LZ>(), 0};
    }
};
// Slots of a column pair's exchanges: the rows of S, all three components (and
// half of them for each parity of a split transform).
template <int LZ> __host__ __device__ constexpr int col_room() { return 3 * (LZ / 2) / (col_split<LZ>() ? 2 : 1); }
template <int LY, int LZ> struct ColMapZ {
    __host__ __device__ static constexpr LaneMap map() {
        return LaneMap{slab_w<LZ>(), 1, slab_w<LZ>(), slab_rs<LY, LZ>(), 1, col_room<LZ>()};
    }
};

// Green tensor for phase B, in the order its threads read it: float4 [hx][pair
// group][idx][3][lane], the pairs (xx, xy), (xz, yy), (yz, zz) of the six
// entries at the point that lane's output idx of that group of column pairs
// stands for (sign of kz included), so that a warp's load is 512 consecutive
// bytes.  The tensors of ky = Ly/2, which share a pair with ky = 0, follow:
// [hx][idx][3][lane of a pair].
template <int LZ> __host__ __device__ constexpr int slab_kz(int idx, int u, int par) {
    constexpr int R = stage_radix<ColPlan<LZ>, -1>(ColPlan<LZ>::NS - 1);
    const int pos = u + (idx / R) * ColPlan<LZ>::NT + (idx % R) * (ColPlan<LZ>::L / R);
    return col_split<LZ>() ? 2 * pos + par : pos;
}
__host__ __device__ constexpr int64_t slab_green_main(int hx, int Ly, int Lz) { return (int64_t)hx * (Ly / 2) * Lz * 3; }
__host__ __device__ constexpr int64_t slab_green_all(int hx, int Ly, int Lz) {
    return slab_green_main(hx, Ly, Lz) + (int64_t)hx * Lz * 3;
}
// from the FP64 octant [6][hz][hy][hx]
template <int LZ>
__global__ void k_slab_green(const double2* __restrict__ gh, float4* __restrict__ out, int hx, int Ly) {
    constexpr int E = ColPlan<LZ>::E, WT = slab_wt<LZ>(), NL = col_lanes<LZ>(), HZ = LZ / 2 + 1;
    const int hy = Ly / 2 + 1, groups = Ly / 2 / WT;
    const int64_t per = (int64_t)hx * hy * HZ, half = slab_green_main(hx, Ly, LZ), total = slab_green_all(hx, Ly, LZ);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t k = i < half ? i : i - half;
        int ky = Ly / 2, lp;  // the pair's ky, and the lane's place in its pair (u + NT par)
        if (i < half) {
            const int lane = (int)(k % 32);
            k /= 32;
            ky = col_pair<LZ>(lane);
            lp = col_lane<LZ>(lane);
        } else {
            lp = (int)(k % NL);
            k /= NL;
        }
        const int q = (int)(k % 3);
        k /= 3;
        const int idx = (int)(k % E);
        k /= E;
        if (i < half) {
            ky += (int)(k % groups) * WT;
            k /= groups;
        }
        const int kx = (int)k, kz = slab_kz<LZ>(idx, lp % ColPlan<LZ>::NT, lp / ColPlan<LZ>::NT);
        const bool fz = kz > LZ / 2;
        const int64_t at = ((int64_t)(fz ? LZ - kz : kz) * hy + ky) * hx + kx;
        const double2 a = gh[2 * q * per + at], b = gh[(2 * q + 1) * per + at];
        // xz (first of the second pair) and yz (first of the third) are odd in z
        const float sa = fz && q > 0 ? -1.f : 1.f;
        out[i] = make_float4(sa * (float)a.x, sa * (float)a.y, (float)b.x, (float)b.y);
    }
}

__device__ __forceinline__ void slab_product(P2& vx, P2& vy, P2& vz, const float4 (&g)[3], const float4 (&h)[3]) {
    // (h: the second half's entries)
    const f32x2 xxr = pk(g[0].x, h[0].x), xxi = pk(g[0].y, h[0].y), xyr = pk(g[0].z, h[0].z), xyi = pk(g[0].w, h[0].w);
    const f32x2 xzr = pk(g[1].x, h[1].x), xzi = pk(g[1].y, h[1].y), yyr = pk(g[1].z, h[1].z), yyi = pk(g[1].w, h[1].w);
    const f32x2 yzr = pk(g[2].x, h[2].x), yzi = pk(g[2].y, h[2].y), zzr = pk(g[2].z, h[2].z), zzi = pk(g[2].w, h[2].w);
    const f32x2 m1 = pk(-1.f, -1.f);
    const P2 a = vx, b = vy, c = vz;
    const f32x2 na = mul2(a.im, m1), nb = mul2(b.im, m1), nc = mul2(c.im, m1);
    vx.re = fma2(xxr, a.re, fma2(xxi, na, fma2(xyr, b.re, fma2(xyi, nb, fma2(xzr, c.re, mul2(xzi, nc))))));
    vx.im = fma2(xxr, a.im, fma2(xxi, a.re, fma2(xyr, b.im, fma2(xyi, b.re, fma2(xzr, c.im, mul2(xzi, c.re))))));
    vy.re = fma2(xyr, a.re, fma2(xyi, na, fma2(yyr, b.re, fma2(yyi, nb, fma2(yzr, c.re, mul2(yzi, nc))))));
    vy.im = fma2(xyr, a.im, fma2(xyi, a.re, fma2(yyr, b.im, fma2(yyi, b.re, fma2(yzr, c.im, mul2(yzi, c.re))))));
    vz.re = fma2(xzr, a.re, fma2(xzi, na, fma2(yzr, b.re, fma2(yzi, nb, fma2(zzr, c.re, mul2(zzi, nc))))));
    vz.im = fma2(xzr, a.im, fma2(xzi, a.re, fma2(yzr, b.im, fma2(yzi, b.re, fma2(zzr, c.im, mul2(zzi, c.re))))));
}

// v[c][idx] *= exp(DIR i pi j / n) at the positions j of a first forward (DIR
// -1) or last inverse (+1) butterfly; tw[j] = exp(-i pi j / n).
template <class PL, int DIR> __device__ __forceinline__ void split_twist(P2 (&v)[3][PL::E], int u, const float2* tw) {
    constexpr int R = DIR < 0 ? stage_radix<PL, -1>(0) : stage_radix<PL, +1>(PL::NS - 1);
#pragma unroll
    for (int q = 0; q < PL::E / R; ++q)
#pragma unroll
        for (int j = 0; j < R; ++j) {
            float2 w = tw[u + q * PL::NT + j * (PL::L / R)];
            if constexpr (DIR > 0) w.y = -w.y;
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c][q * R + j] = pmul(v[c][q * R + j], pk(w.x, w.x), pk(w.y, w.y), pk(-w.y, -w.y));
        }
}

template <int LY, int LZ, int NB>
__global__ void __launch_bounds__(slab_threads<LY, LZ, NB>(), NB)
    k_slab(float2* __restrict__ U, const float4* __restrict__ G, int Lx, const float2* __restrict__ twy,
           const float2* __restrict__ twz, const int* __restrict__ active) {
    using PY = RowPlan<LY>;
    using PZ = ColPlan<LZ>;
    constexpr int NY = LY / 2, NZ = LZ / 2, RS = slab_rs<LY, LZ>(), RH = NZ / 2 * RS;
    constexpr int NTH = slab_threads<LY, LZ, NB>(), NW = NTH / 32, WT = slab_wt<LZ>();
    static_assert(NTH % 32 == 0 && (LY / 2) % WT == 0, "whole warps and whole pair groups");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* S = reinterpret_cast<float2*>(smem_raw);
    float2 *tyf = S + 3 * NZ * RS, *tyi = tyf + LY, *tzf = tyi + LY, *tzi = tzf + PZ::L, *tzs = tzi + PZ::L;
    static_assert(pair_tw_size<PY, -1>() <= LY && pair_tw_size<PY, 1>() <= LY, "twiddle tables");
    static_assert(pair_tw_size<PZ, -1>() <= PZ::L && pair_tw_size<PZ, 1>() <= PZ::L, "twiddle tables");
    const int kx = blockIdx.x, r = blockIdx.y;
    if (active != nullptr && active[r] == 0) return;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int64_t cstride = (int64_t)Lx * NZ * NY;
    float2* ub = U + (int64_t)r * 3 * cstride + (int64_t)kx * NZ * NY;
    pair_tw_fill<PY, -1>(tyf, twy, threadIdx.x, NTH);
    pair_tw_fill<PY, +1>(tyi, twy, threadIdx.x, NTH);
    // the slab's rows, 16 bytes per thread and copy, all in flight at once
    constexpr int CPR = NY / 2;  // copies per row
    for (int e = threadIdx.x; e < 3 * NZ * CPR; e += NTH) {
        const int row = e / CPR, o = e - row * CPR, c = row / NZ;
        const float2* src = ub + c * cstride + (row - c * NZ) * NY + 2 * o;
        const unsigned dst = (unsigned)__cvta_generic_to_shared(S + row * RS + 2 * o);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    }
    constexpr int ZS = LZ / PZ::L;  // (2 where the transform is split)
    pair_tw_fill<PZ, -1>(tzf, twz, threadIdx.x, NTH, ZS);
    pair_tw_fill<PZ, +1>(tzi, twz, threadIdx.x, NTH, ZS);
    if constexpr (ZS > 1)
        for (int e = threadIdx.x; e < NZ; e += NTH) tzs[e] = twz[e];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const bool fx = kx > Lx / 2;
    constexpr int RPW = 32 / PY::NT, NRP = 3 * NZ / 2;  // row pairs of a warp, of the slab
    // ---- A: rows forward
    {
        constexpr int E = PY::E, NT = PY::NT, R0 = stage_radix<PY, -1>(0), NB0 = E / R0;
        const int p = lane / NT, u = lane % NT;
#pragma unroll 1
        for (int g = warp; g * RPW < NRP; g += NW) {
            const int rp = min(g * RPW + p, NRP - 1);
            const bool ok = g * RPW + p < NRP;
            const int c = rp / (NZ / 2), iz = slab_row<LY, LZ>(rp - c * (NZ / 2));
            const float sg = (fx && c == 0) ? -1.f : 1.f;
            f32x2* row = reinterpret_cast<f32x2*>(S + (c * NZ + iz) * RS);
            P2 v[1][E];
#pragma unroll
            for (int q = 0; q < NB0; ++q)
#pragma unroll
                for (int j = 0; j < R0 / 2; ++j) {
                    const int pos = u + q * NT + j * (LY / R0);
                    const float2 a = upk(row[pos]), b = upk(row[RH + pos]);
                    v[0][q * R0 + j] = P2{pk(sg * a.x, sg * b.x), pk(sg * a.y, sg * b.y)};
                }
            auto st = [&](int s, P2 x) {
                if (ok) {
                    row[s] = x.re;
                    row[RH + s] = x.im;
                }
            };
            auto ld = [&](int s) { return P2{row[s], row[RH + s]}; };
            pair_stages<PY, -1, 0, 1, RowMapY<LY, LZ>>(v, u, tyf, ld, st, true);
            __syncwarp();
            if (ok)
                for_each_out<PY, -1, false>(u, [&](int idx, int pos) {
                    const float2 re = upk(v[0][idx].re), im = upk(v[0][idx].im);
                    reinterpret_cast<float2*>(row)[pos] = make_float2(re.x, im.x);
                    reinterpret_cast<float2*>(row)[RH + pos] = make_float2(re.y, im.y);
                });
        }
    }
    __syncthreads();
    // ---- B: columns
    {
        constexpr int E = PZ::E, NT = PZ::NT, R0 = stage_radix<PZ, -1>(0), NB0 = E / R0;
        constexpr bool SPLIT = col_split<LZ>();
        constexpr int JN = SPLIT ? R0 : R0 / 2;  // inputs of a first butterfly: all of the split's n, half of Lz
        const int t = col_pair<LZ>(lane), u = col_lane<LZ>(lane) % NT, par = col_lane<LZ>(lane) / NT;
        const int kxo = fx ? Lx - kx : kx;
        const float4* gx = G + (int64_t)kxo * (LY / 2) * LZ * 3 + lane;
        const float4* g0 = G + slab_green_main(Lx / 2 + 1, LY, LZ) + (int64_t)kxo * LZ * 3 + col_lane<LZ>(lane);
#pragma unroll 1
        for (int g = warp; g * WT < LY / 2; g += NW) {
            const int k0 = g * WT + t, k1 = k0 == 0 ? LY / 2 : LY - k0;
            P2 v[3][E];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int q = 0; q < NB0; ++q)
#pragma unroll
                    for (int j = 0; j < JN; ++j) {
                        const float2* row = S + (c * NZ + u + q * NT + j * (PZ::L / R0)) * RS;
                        const float2 a = row[k0];
                        float2 b = row[k1];
                        if (c == 1) b = make_float2(-b.x, -b.y);
                        v[c][q * R0 + j] = P2{pk(a.x, b.x), pk(a.y, b.y)};
                    }
            if constexpr (SPLIT) {  // the odd frequencies' inputs (DIR -1) and outputs (+1) carry exp(-+i pi j / n)
                if (par) split_twist<PZ, -1>(v, u, tzs);
            }
            // exchange words: slot s is row s of S, real parts in column k0 and
            // imaginary parts in k1 (split: the odd parity takes the upper rows)
            f32x2* s0 = reinterpret_cast<f32x2*>(S) + k0 + par * (col_room<LZ>() * RS);
            f32x2* s1 = s0 + (k1 - k0);
            auto st = [&](int s, P2 x) {
                s0[s * RS] = x.re;
                s1[s * RS] = x.im;
            };
            auto ld = [&](int s) { return P2{s0[s * RS], s1[s * RS]}; };
            pair_stages<PZ, -1, 0, 3, ColMapZ<LY, LZ>>(v, u, tzf, ld, st, !SPLIT);
            // (group 0 holds the pair of the two self-mirrored columns, which
            // have a tensor each)
            if (g != 0) {
#pragma unroll
                for (int idx = 0; idx < E; ++idx) {
                    float4 ga[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) ga[i] = __ldg(gx + ((g * E + idx) * 3 + i) * 32);
                    slab_product(v[0][idx], v[1][idx], v[2][idx], ga, ga);
                }
            } else {
#pragma unroll
                for (int idx = 0; idx < E; ++idx) {
                    float4 ga[3], gb[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) ga[i] = __ldg(gx + (idx * 3 + i) * 32);
#pragma unroll
                    for (int i = 0; i < 3; ++i) gb[i] = t == 0 ? __ldg(g0 + (idx * 3 + i) * col_lanes<LZ>()) : ga[i];
                    slab_product(v[0][idx], v[1][idx], v[2][idx], ga, gb);
                }
            }
            pair_stages<PZ, +1, 0, 3, ColMapZ<LY, LZ>>(v, u, tzi, ld, st, false);
            __syncwarp();
            auto put = [&](int c, int pos, P2 x) {
                const float2 re = upk(x.re), im = upk(x.im);
                float2* row = S + (c * NZ + pos) * RS;
                row[k0] = make_float2(re.x, im.x);
                row[k1] = c == 1 ? make_float2(-re.y, -im.y) : make_float2(re.y, im.y);
            };
            if constexpr (!SPLIT) {
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    for_each_out<PZ, +1, true>(u, [&](int idx, int pos) { put(c, pos, v[c][idx]); });
            } else {
                if (par) split_twist<PZ, +1>(v, u, tzs);
                // each lane of the two adds and stores half of the outputs
                constexpr int RI = stage_radix<PZ, +1>(PZ::NS - 1);
                static_assert(E == RI, "one butterfly per thread");
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int m = 0; m < RI / 2; ++m) {
                        const P2 lo = v[c][m], hi = v[c][m + RI / 2];
                        const P2 send = par ? lo : hi, keep = par ? hi : lo;
                        const P2 got{__shfl_xor_sync(0xffffffffu, send.re, 16), __shfl_xor_sync(0xffffffffu, send.im, 16)};
                        put(c, u + (m + (par ? RI / 2 : 0)) * NT, padd(keep, got));
                    }
            }
        }
    }
    __syncthreads();
    // ---- C: rows inverse
    {
        constexpr int E = PY::E, NT = PY::NT, R0 = stage_radix<PY, +1>(0), NB0 = E / R0;
        const int p = lane / NT, u = lane % NT;
#pragma unroll 1
        for (int g = warp; g * RPW < NRP; g += NW) {
            const int rp = min(g * RPW + p, NRP - 1);
            const bool ok = g * RPW + p < NRP;
            const int c = rp / (NZ / 2), iz = slab_row<LY, LZ>(rp - c * (NZ / 2));
            const float sg = (fx && c == 0) ? -1.f : 1.f;
            f32x2* row = reinterpret_cast<f32x2*>(S + (c * NZ + iz) * RS);
            P2 v[1][E];
#pragma unroll
            for (int q = 0; q < NB0; ++q)
#pragma unroll
                for (int j = 0; j < R0; ++j) {
                    const int pos = u + q * NT + j * (LY / R0);
                    const float2 a = reinterpret_cast<float2*>(row)[pos], b = reinterpret_cast<float2*>(row)[RH + pos];
                    v[0][q * R0 + j] = P2{pk(a.x, b.x), pk(a.y, b.y)};
                }
            auto st = [&](int s, P2 x) {
                if (ok) {
                    row[s] = x.re;
                    row[RH + s] = x.im;
                }
            };
            auto ld = [&](int s) { return P2{row[s], row[RH + s]}; };
            pair_stages<PY, +1, 0, 1, RowMapY<LY, LZ>>(v, u, tyi, ld, st, false);
            __syncwarp();
            if (ok)
                for_each_out<PY, +1, true>(u, [&](int idx, int pos) {
                    const float2 re = upk(v[0][idx].re), im = upk(v[0][idx].im);
                    reinterpret_cast<float2*>(row)[pos] = make_float2(sg * re.x, sg * im.x);
                    reinterpret_cast<float2*>(row)[RH + pos] = make_float2(sg * re.y, sg * im.y);
                });
            // the finished rows leave by bulk copies, one per row
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (ok && u < 2) {
                const unsigned src = (unsigned)__cvta_generic_to_shared(row + u * RH);
                float2* out = ub + c * cstride + (iz + u * (NZ / 2)) * NY;
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out), "r"(src),
                             "r"((unsigned)(NY * 8))
                             : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        // (shared memory must outlive the copies out of it)
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
}

template <int LY, int LZ>
cudaError_t launch_slab(const Geom& g, int R, float2* u, const float4* gs, const Twiddles<float>& tw, const int* active,
                        cudaStream_t st) {
    constexpr size_t sm = slab_smem<LY, LZ>();
    static_assert(sm <= 227 * 1024, "the slab does not fit in shared memory");
    // 152 SMs: with at most one slab each, a slab takes all of an SM's threads
    // (32^3 lattice, one RHS, 64 slabs: see slab_threads)
    constexpr int NB = slab_blocks<LY, LZ>();
    const bool wide = NB > 1 && (int64_t)g.Lx * R <= 152;
    auto kern = wide ? k_slab<LY, LZ, 1> : k_slab<LY, LZ, NB>;
    const int threads = wide ? slab_threads<LY, LZ, 1>() : slab_threads<LY, LZ, NB>();
    cudaError_t e = allow_smem(kern, sm);
    if (e != cudaSuccess) return e;
    PROF_BEGIN(st);
    kern<<<dim3(g.Lx, R), threads, sm, st>>>(u, gs, g.Lx, tw.y, tw.z, active);
    PROF_END(KK_SLAB_C64, R, st);
    return cudaGetLastError();
}

}  // namespace dda

// slab_fn_<LY>: the launchers of one y length (its own translation unit).
#define DDA_SLAB_DEFINE(LY)                                \
    namespace dda {                                        \
    DDA_SLAB_FN(LY) {                                      \
        switch (Lz) {                                      \
            case 16: return launch_slab<LY, 16>;           \
            case 32: return launch_slab<LY, 32>;           \
            case 48: return launch_slab<LY, 48>;           \
            case 64: return launch_slab<LY, 64>;           \
            case 96: return launch_slab<LY, 96>;           \
            case 128: return launch_slab<LY, 128>;         \
            default: return nullptr;                       \
        }                                                  \
    }                                                      \
    }
