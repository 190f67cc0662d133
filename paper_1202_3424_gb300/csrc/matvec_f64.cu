// complex128 instantiation of the matvec passes, the Green-tensor build and shared host helpers.
#include <algorithm>

#include "matvec_impl.cuh"

namespace dda {

template int zconv_schedules<double>(const Geom&);
template int xpass_schedules<double>(const Geom&);
template int ypass_schedules<double>(const Geom&);
template cudaError_t launch_zconv<double>(const Geom&, int, double2*, const double2*, const double2*, const int*, int, cudaStream_t);
template cudaError_t launch_matvec<double>(const Geom&, int, const double2*, double2*, const PadWork<double>&,
                                           const DevTarget&, const double2*, int, const double2*,
                                           const Twiddles<double>&, const int*, cudaStream_t);
template cudaError_t launch_matvec_fused<double>(const Geom&, int, double2*, double2*, const PadWork<double>&,
                                                 const DevTarget&, const double2*, int, const double2*,
                                                 const Twiddles<double>&, int*, const FusedKrylov<double>&,
                                                 cudaStream_t);

int pick_fft_length(int n) {
    for (int L : kSupportedLengths)
        if (L >= 2 * n) return L;
    return 0;
}

// Blocks of one RHS in the x-inverse pass (partial-sum slots per RHS): the
// most among the staged tilings of complex64 and 16-byte elements and the
// warp-local blocks of every plan variant.
template <int L, int V = 0> static int min_xwi_rows() {
    int tp = xwi_rows<XwPlan<L, V>>();
    if constexpr (V + 1 < xw_variants(L)) {
        const int rest = min_xwi_rows<L, V + 1>();
        tp = rest < tp ? rest : tp;
    }
    return tp;
}
template <int L> static int min_tp_x() {
    int tp = tp_x<L, 8>() < tp_x<L, 16>() ? tp_x<L, 8>() : tp_x<L, 16>();
    return min_xwi_rows<L>() < tp ? min_xwi_rows<L>() : tp;
}
int xinv_blocks_per_rhs(const Geom& g) {
    const int nrows = g.ny * g.nz;
    int tp = 1;
    switch (g.Lx) {
        case 16: tp = min_tp_x<16>(); break;
        case 32: tp = min_tp_x<32>(); break;
        case 48: tp = min_tp_x<48>(); break;
        case 64: tp = min_tp_x<64>(); break;
        case 96: tp = min_tp_x<96>(); break;
        case 128: tp = min_tp_x<128>(); break;
        case 192: tp = min_tp_x<192>(); break;
        case 256: tp = min_tp_x<256>(); break;
        case 384: tp = min_tp_x<384>(); break;
        case 512: tp = min_tp_x<512>(); break;
        default: tp = 1;
    }
    return 3 * ((nrows + tp - 1) / tp);
}

// ---- Green tensor ---------------------------------------------------------------
// Every component is even or odd under each axis reflection, and so is its
// transform, of which only the octant k <= L/2 is kept.  So one octant of the
// displacements is formed, and along each axis the lines of the octants already
// transformed and not yet transformed are mirrored as they are loaded: a quarter
// of the lines of the full padded grid per axis, an eighth of its points.  (The
// transforms are FP64-bound: 192^3 padded, 7.6 -> 1.9 ms for the four kernels,
// and 0.7 GB of scratch -> 0.17 GB; the results keep their bits.)

// xx, xy, xz, yy, yz, zz: odd in x (axis 0), y (1), z (2)?
__host__ __device__ constexpr bool green_odd(int c, int axis) {
    return axis == 0 ? (c == 1 || c == 2) : (axis == 1 ? (c == 1 || c == 4) : (c == 2 || c == 4));
}

// A(r) = exp(ik rho)/rho [k^2 (rr - I) + (ik rho - 1)/rho^2 (3 rr - I)]
// (Draine 1988 off-diagonal block, lattice units), components xx,xy,xz,yy,yz,zz,
// at the displacements 0 <= d < n per axis (zero at r = 0): g [6][nz][ny][nx].
__global__ void k_green(double2* __restrict__ g, int nx, int ny, int nz, double kd) {
    const int64_t total = (int64_t)nx * ny * nz;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int dx = (int)(idx % nx), dy = (int)((idx / nx) % ny), dz = (int)(idx / ((int64_t)nx * ny));
        double2 a[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) a[c] = make_double2(0.0, 0.0);
        if ((dx | dy | dz) != 0) {
            const double rho2 = (double)dx * dx + (double)dy * dy + (double)dz * dz;
            const double rho = sqrt(rho2);
            const double rh[3] = {dx / rho, dy / rho, dz / rho};
            double sn, cs;
            sincos(kd * rho, &sn, &cs);
            const double2 ph = make_double2(cs / rho, sn / rho);             // exp(ik rho)/rho
            const double2 c1 = make_double2(kd * kd * ph.x, kd * kd * ph.y);  // k^2 ph
            const double2 t = make_double2(-1.0 / rho2, kd / rho);           // (ik rho - 1)/rho^2
            const double2 c2 = cmul(ph, t);
            const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const double rr = rh[ia[c]] * rh[ib[c]];
                const double dl = ia[c] == ib[c] ? 1.0 : 0.0;
                const double f1 = rr - dl, f2 = 3.0 * rr - dl;
                a[c] = make_double2(c1.x * f1 + c2.x * f2, c1.y * f1 + c2.y * f2);
            }
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) g[c * total + idx] = a[c];
    }
}

// x lines: rows [LX/2] of src, mirrored to LX points, transformed; the LX/2 + 1
// frequencies of the octant to dst.  blockIdx.y: component.
template <int LX>
__global__ void __launch_bounds__(tp_x<LX, 16>() * Plan<LX>::NT)
    k_green_x(const double2* __restrict__ src, double2* __restrict__ dst, int nrows, const double2* __restrict__ tw) {
    using C = double2;
    using PL = Plan<LX>;
    constexpr int TP = tp_x<LX, 16>(), SP = TP + 1, NX = LX / 2, HX = LX / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int c = blockIdx.y, row0 = blockIdx.x * TP;
    const double sg = green_odd(c, 0) ? -1.0 : 1.0;
    src += (int64_t)c * nrows * NX;
    dst += (int64_t)c * nrows * HX;
    for (int e = threadIdx.x; e < TP * NX; e += blockDim.x) {
        const int t2 = e / NX, x = e - t2 * NX, row = row0 + t2;
        const C v = row < nrows ? src[(int64_t)row * NX + x] : czero<C>();
        buf[x * SP + t2] = v;
        buf[(x == 0 ? NX : LX - x) * SP + t2] = x == 0 ? czero<C>() : cscale(v, sg);
    }
    __syncthreads();
    const int t = threadIdx.x % TP, u = threadIdx.x / TP;
    C* bt = buf + t;
    C v[PL::E];
    auto first = [&](int pos) { return bt[pos * SP]; };
    auto ld = [&](int pos) { return bt[pos * SP]; };
    auto st = [&](int pos, C val) { bt[pos * SP] = val; };
    pencil_fft<C, PL, -1, false>(v, u, tw, first, ld, st);
    __syncthreads();
    for_each_out<PL, -1, false>(u, [&](int idx, int pos) { bt[pos * SP] = v[idx]; });
    __syncthreads();
    for (int e = threadIdx.x; e < TP * HX; e += blockDim.x) {
        const int t2 = e / HX, x = e - t2 * HX, row = row0 + t2;
        if (row < nrows) dst[(int64_t)row * HX + x] = buf[x * SP + t2];
    }
}

// y and z lines: `width` adjacent lines of L/2 points pt apart, mirrored, the
// L/2 + 1 frequencies of the octant (times scale) to dst with the same point
// stride.  blockIdx.y: component * batches + batch.
template <int L>
__global__ void __launch_bounds__(tp_sp<SPlan<L, 0>, 16>() * SPlan<L, 0>::NT)
    k_green_line(const double2* __restrict__ src, double2* __restrict__ dst, int64_t pt, int width, int batches,
                 int axis, double scale, const double2* __restrict__ tw) {
    using C = double2;
    using PL = SPlan<L, 0>;
    constexpr int TP = tp_sp<PL, 16>(), N = L / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int b = blockIdx.y, t = threadIdx.x % TP, u = threadIdx.x / TP, w = blockIdx.x * TP + t;
    const bool valid = w < width;
    const double sg = green_odd(b / batches, axis) ? -1.0 : 1.0;
    const C* s = src + (int64_t)b * N * pt + (valid ? w : 0);
    C* d = dst + (int64_t)b * (N + 1) * pt + (valid ? w : 0);
    C* bt = buf + t;
    C v[PL::E];
    auto first = [&](int pos) {
        if (!valid || pos == N) return czero<C>();
        return pos < N ? s[pos * pt] : cscale(s[(L - pos) * pt], sg);
    };
    auto ld = [&](int pos) { return bt[pos * TP]; };
    auto st = [&](int pos, C val) { bt[pos * TP] = val; };
    pencil_fft<C, PL, -1, false>(v, u, tw, first, ld, st);
    for_each_out<PL, -1, false>(u, [&](int idx, int pos) {
        if (valid && pos <= N) d[pos * pt] = cscale(v[idx], scale);
    });
}

__global__ void k_c128_to_c64(const double2* __restrict__ s, float2* __restrict__ d, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = make_float2((float)s[i].x, (float)s[i].y);
}

template <typename D, typename S>
__global__ void k_cconvert(const S* __restrict__ s, D* __restrict__ d, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = ccast<D>(s[i]);
}

template <int LX>
static cudaError_t green_x(const double2* src, double2* dst, int nrows, const double2* tw, cudaStream_t st) {
    constexpr int TP = tp_x<LX, 16>(), NTH = TP * Plan<LX>::NT;
    const size_t sm = (size_t)LX * (TP + 1) * sizeof(double2);
    cudaError_t e = allow_smem(k_green_x<LX>, sm);
    if (e != cudaSuccess) return e;
    PROF_BEGIN(st);
    k_green_x<LX><<<dim3((nrows + TP - 1) / TP, 6), NTH, sm, st>>>(src, dst, nrows, tw);
    PROF_END(KK_GREEN, 1.0, st);
    return cudaGetLastError();
}
template <int L>
static cudaError_t green_line(const double2* src, double2* dst, int64_t pt, int width, int batches, int axis,
                              double scale, const double2* tw, cudaStream_t st) {
    using PL = SPlan<L, 0>;
    constexpr int TP = tp_sp<PL, 16>(), NTH = TP * PL::NT;
    const size_t sm = (size_t)L * TP * sizeof(double2);
    cudaError_t e = allow_smem(k_green_line<L>, sm);
    if (e != cudaSuccess) return e;
    PROF_BEGIN(st);
    k_green_line<L><<<dim3((width + TP - 1) / TP, 6 * batches), NTH, sm, st>>>(src, dst, pt, width, batches, axis,
                                                                              scale, tw);
    PROF_END(KK_GREEN, 1.0, st);
    return cudaGetLastError();
}

// Two buffers: the octant of displacements (and, once that is transformed
// along x, the y-transformed octant), and the x-transformed one.
static int64_t green_a(const Geom& g) { return 6 * std::max((int64_t)g.nx * g.ny * g.nz, (int64_t)g.hx() * g.hy() * g.nz); }
int64_t green_scratch_size(const Geom& g) { return green_a(g) + 6 * (int64_t)g.hx() * g.ny * g.nz; }

cudaError_t launch_green_fft(const Geom& g, double kd, double2* scratch, double2* ghat64, const Twiddles<double>& tw,
                             cudaStream_t st) {
    double2 *a = scratch, *b = scratch + green_a(g);
    const int hx = g.hx(), hy = g.hy();
    PROF_BEGIN(st);
    k_green<<<grid1d((int64_t)g.nx * g.ny * g.nz, 256), 256, 0, st>>>(a, g.nx, g.ny, g.nz, kd);
    PROF_END(KK_GREEN, 1.0, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    auto xf = [&]() -> cudaError_t { DDA_DISPATCH_L(g.Lx, green_x, a, b, g.ny * g.nz, tw.x, st); };
    if ((e = xf()) != cudaSuccess) return e;
    auto yf = [&]() -> cudaError_t { DDA_DISPATCH_L(g.Ly, green_line, b, a, (int64_t)hx, hx, g.nz, 1, 1.0, tw.y, st); };
    if ((e = yf()) != cudaSuccess) return e;
    const double scale = 1.0 / ((double)g.Lx * g.Ly * g.Lz);
    auto zf = [&]() -> cudaError_t {
        DDA_DISPATCH_L(g.Lz, green_line, a, ghat64, (int64_t)hx * hy, hx * hy, 1, 2, scale, tw.z, st);
    };
    return zf();
}

cudaError_t launch_convert_c128_to_df(const double2* src, cdfl* dst, int64_t n, cudaStream_t st) {
    k_cconvert<cdfl, double2><<<grid1d(n, 256), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_convert_df_to_c128(const cdfl* src, double2* dst, int64_t n, cudaStream_t st) {
    k_cconvert<double2, cdfl><<<grid1d(n, 256), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_convert_c128_to_c64(const double2* src, float2* dst, int64_t n, cudaStream_t st) {
    k_c128_to_c64<<<grid1d(n, 256), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}



}  // namespace dda
