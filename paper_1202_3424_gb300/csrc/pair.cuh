// FFT pencils in packed FP32 pairs.
//
// The FP32 pipes of sm_103a take two operations per instruction when both
// operands are pairs of registers (add, sub, mul, fma .f32x2): the same
// operations per clock as the scalar instructions (measured: 37 T/s each
// way), for half the issue slots.  An FFT pass issues shared-memory and
// address instructions between its arithmetic, so with scalar arithmetic it
// stops at the issue rate with the FP32 pipes half idle.  Here one thread
// runs two pencils in lockstep, one in each half of every pair: all radix
// stages are the same for both, so every arithmetic instruction serves two
// points.  Real and imaginary parts sit in pairs of their own (P2), so that
// a product with a shared twiddle needs no shuffling of halves, and a product
// with +-i is a change of name plus the sign of an addition.
#pragma once

#include "fft.cuh"

namespace dda {

// Two complex numbers, one per half.
struct P2 {
    f32x2 re, im;
};
__device__ __forceinline__ P2 padd(P2 a, P2 b) { return P2{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ P2 psub(P2 a, P2 b) { return P2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a + SGN i b
template <int SGN> __device__ __forceinline__ P2 padd_i(P2 a, P2 b) {
    if constexpr (SGN > 0) return P2{sub2(a.re, b.im), add2(a.im, b.re)};
    else return P2{add2(a.re, b.im), sub2(a.im, b.re)};
}
// e + s q for a real scalar pair s
__device__ __forceinline__ P2 pfma(P2 q, f32x2 s, P2 e) { return P2{fma2(q.re, s, e.re), fma2(q.im, s, e.im)}; }
// a (c + i y), with ny = -y
__device__ __forceinline__ P2 pmul(P2 a, f32x2 c, f32x2 y, f32x2 ny) {
    return P2{fma2(a.im, ny, mul2(a.re, c)), fma2(a.im, c, mul2(a.re, y))};
}

// ---- small DFTs, sign convention exp(SGN * 2 pi i j k / R) ----------------
template <int R, int SGN> struct PDft;

template <int SGN> struct PDft<3, SGN> {
    __device__ __forceinline__ static void run(P2* v) {
        const f32x2 h = pk(-0.5f, -0.5f);
        const float s3 = SGN * 0.86602540378443864676f;  // sin(pi/3)
        const f32x2 s = pk(s3, s3), ns = pk(-s3, -s3);
        const P2 t = padd(v[1], v[2]), d = psub(v[1], v[2]);
        const P2 m = pfma(t, h, v[0]);
        v[0] = padd(v[0], t);
        v[1] = P2{fma2(d.im, ns, m.re), fma2(d.re, s, m.im)};
        v[2] = P2{fma2(d.im, s, m.re), fma2(d.re, ns, m.im)};
    }
};

template <int SGN> struct PDft<4, SGN> {
    __device__ __forceinline__ static void run(P2* v) {
        const P2 t0 = padd(v[0], v[2]), t1 = psub(v[0], v[2]);
        const P2 t2 = padd(v[1], v[3]), d = psub(v[1], v[3]);
        v[0] = padd(t0, t2);
        v[2] = psub(t0, t2);
        v[1] = padd_i<SGN>(t1, d);
        v[3] = padd_i<-SGN>(t1, d);
    }
    // inputs 2 and 3 are zero
    __device__ __forceinline__ static void run_half(P2* v) {
        const P2 a = v[0], b = v[1];
        v[0] = padd(a, b);
        v[2] = psub(a, b);
        v[1] = padd_i<SGN>(a, b);
        v[3] = padd_i<-SGN>(a, b);
    }
};

// Radix 6 as 2 x 3: the DFTs of the even and odd inputs, then the twiddles
// w6^k (w6^1 = (1 + SGN i sqrt3)/2, w6^2 = (-1 + SGN i sqrt3)/2).
template <int SGN> struct PDft<6, SGN> {
    __device__ __forceinline__ static void run(P2* v) {
        P2 e[3] = {v[0], v[2], v[4]};
        P2 o[3] = {v[1], v[3], v[5]};
        PDft<3, SGN>::run(e);
        PDft<3, SGN>::run(o);
        const float s3 = SGN * 0.86602540378443864676f;
        const f32x2 h = pk(0.5f, 0.5f), nh = pk(-0.5f, -0.5f), s = pk(s3, s3), ns = pk(-s3, -s3);
        o[1] = pmul(o[1], h, s, ns);
        o[2] = pmul(o[2], nh, s, ns);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            v[k] = padd(e[k], o[k]);
            v[k + 3] = psub(e[k], o[k]);
        }
    }
};

template <int SGN> struct PDft<8, SGN> {
    __device__ __forceinline__ static void combine(P2* v, P2 (&e)[4], P2 (&o)[4]) {
        const f32x2 r2 = pk(0.70710678118654752440f, 0.70710678118654752440f);
        const f32x2 nr2 = pk(-0.70710678118654752440f, -0.70710678118654752440f);
        // w8^1 = (1 + SGN i)/sqrt2, w8^2 = SGN i, w8^3 = -(1 - SGN i)/sqrt2
        const P2 q1 = padd_i<SGN>(o[1], o[1]), q3 = padd_i<-SGN>(o[3], o[3]);
        v[0] = padd(e[0], o[0]);
        v[4] = psub(e[0], o[0]);
        v[1] = pfma(q1, r2, e[1]);
        v[5] = pfma(q1, nr2, e[1]);
        v[2] = padd_i<SGN>(e[2], o[2]);
        v[6] = padd_i<-SGN>(e[2], o[2]);
        v[3] = pfma(q3, nr2, e[3]);
        v[7] = pfma(q3, r2, e[3]);
    }
    __device__ __forceinline__ static void run(P2* v) {
        P2 e[4] = {v[0], v[2], v[4], v[6]};
        P2 o[4] = {v[1], v[3], v[5], v[7]};
        PDft<4, SGN>::run(e);
        PDft<4, SGN>::run(o);
        combine(v, e, o);
    }
    // inputs 4..7 are zero
    __device__ __forceinline__ static void run_half(P2* v) {
        P2 e[4] = {v[0], v[2], v[0], v[0]};
        P2 o[4] = {v[1], v[3], v[1], v[1]};
        PDft<4, SGN>::run_half(e);
        PDft<4, SGN>::run_half(o);
        combine(v, e, o);
    }
};

// Radix 16 as 4 x 4: n = 4 n1 + n2, k = k1 + 4 k2.
template <int SGN> struct PDft<16, SGN> {
    template <int J> __device__ __forceinline__ static P2 w16(P2 a) {
        const float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, r2 = 0.70710678118654752440f;
        if constexpr (J == 1) return pmul(a, pk(c1, c1), pk(SGN * s1, SGN * s1), pk(-SGN * s1, -SGN * s1));
        else if constexpr (J == 3) return pmul(a, pk(s1, s1), pk(SGN * c1, SGN * c1), pk(-SGN * c1, -SGN * c1));
        else if constexpr (J == 9) return pmul(a, pk(-c1, -c1), pk(-SGN * s1, -SGN * s1), pk(SGN * s1, SGN * s1));
        else if constexpr (J == 2) {
            const P2 q = padd_i<SGN>(a, a);
            return P2{mul2(q.re, pk(r2, r2)), mul2(q.im, pk(r2, r2))};
        } else {  // J == 6: (-1 + SGN i)/sqrt2
            const P2 q = padd_i<-SGN>(a, a);
            return P2{mul2(q.re, pk(-r2, -r2)), mul2(q.im, pk(-r2, -r2))};
        }
    }
    __device__ __forceinline__ static void run(P2* v) {
        P2 y[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < 4; ++n1) y[n2][n1] = v[4 * n1 + n2];
            PDft<4, SGN>::run(y[n2]);
        }
        // (the product with w16^4 = SGN i of y[2][2] goes into the last DFT's sums)
        y[1][1] = w16<1>(y[1][1]);
        y[1][2] = w16<2>(y[1][2]);
        y[1][3] = w16<3>(y[1][3]);
        y[2][1] = w16<2>(y[2][1]);
        y[2][3] = w16<6>(y[2][3]);
        y[3][1] = w16<3>(y[3][1]);
        y[3][2] = w16<6>(y[3][2]);
        y[3][3] = w16<9>(y[3][3]);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            P2 z[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
            if (k1 == 2) {
                const P2 t0 = padd_i<SGN>(z[0], z[2]), t1 = padd_i<-SGN>(z[0], z[2]);
                const P2 t2 = padd(z[1], z[3]), d = psub(z[1], z[3]);
                z[0] = padd(t0, t2);
                z[2] = psub(t0, t2);
                z[1] = padd_i<SGN>(t1, d);
                z[3] = padd_i<-SGN>(t1, d);
            } else {
                PDft<4, SGN>::run(z);
            }
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = z[k2];
        }
    }
};

// ---- exchange addresses --------------------------------------------------
// The exchanges of a warp go through 8-byte shared-memory words; the 16 lanes
// of a half-warp are served at once when their words lie on 16 different
// banks (word address mod 16).  Two maps from the position exchanged after
// stage S to a slot keep them apart:
//   swizzle  pos ^ ((pos >> K) & 15), which stays inside the aligned block of
//            16, for pencils without a word to spare;
//   padding  pos + (pos >> K), one slot after every 2^K, whose addresses are a
//            per-thread base plus constants (no instruction per access).
// best_key counts the wavefronts of every exchange instruction of a plan for
// each K and takes the cheapest, at compile time.  LaneMap: lane l holds
// thread u = (l / us) % NT of pencil (l / ps) % npen, whose slot s lies on
// bank s * sb + pencil * pb; slots is the room per pencil (0: swizzle).
struct LaneMap {
    int us, ps, npen, sb, pb, slots;
};
template <class PL, int DIR, int S> struct ExchangePos {
    static constexpr int L = PL::L, NT = PL::NT, R = stage_radix<PL, DIR>(S), P = stage_p<PL, DIR>(S),
                         R2 = stage_radix<PL, DIR>(S + 1);
    static constexpr bool kLinear = NT % P == 0;  // store offsets constant across butterflies
    // register k of thread u: the part of its position that depends on u, and the rest
    __host__ __device__ static constexpr int store_base(int u, int k) {
        return kLinear ? (u / P) * (P * R) + u % P : ((u + k / R * NT) / P) * (P * R) + (u + k / R * NT) % P;
    }
    __host__ __device__ static constexpr int store_off(int k) { return (kLinear ? k / R * NT * R : 0) + k % R * P; }
    __host__ __device__ static constexpr int load_off(int k) { return k / R2 * NT + k % R2 * (L / R2); }
};
template <class PL, int DIR, int S> __host__ __device__ constexpr int exchange_cost(LaneMap m, int K) {
    using X = ExchangePos<PL, DIR, S>;
    int cost = 0;
    for (int half = 0; half < 2; ++half)
        for (int k = 0; k < PL::E; ++k)
            for (int load = 0; load < 2; ++load) {
                int seen[16] = {};
                int worst = 0;
                for (int l = half * 16; l < half * 16 + 16; ++l) {
                    const int u = (l / m.us) % PL::NT, pen = (l / m.ps) % m.npen;
                    const int pos = load ? u + X::load_off(k) : X::store_base(u, k) + X::store_off(k);
                    const int slot = K == 0 ? pos : (m.slots ? pos + (pos >> K) : pos ^ ((pos >> K) & 15));
                    const int bank = ((slot * m.sb + pen * m.pb) % 16 + 16) % 16;
                    if (++seen[bank] > worst) worst = seen[bank];
                }
                cost += worst;
            }
    return cost;
}
// padding: base and offset can be padded apart (no carry between them), and the slots suffice
template <class PL, int DIR, int S> __host__ __device__ constexpr bool pad_folds(LaneMap m, int K) {
    using X = ExchangePos<PL, DIR, S>;
    if (PL::L + ((PL::L - 1) >> K) > m.slots) return false;
    for (int u = 0; u < PL::NT; ++u)
        for (int k = 0; k < PL::E; ++k) {
            const int mask = (1 << K) - 1;
            if ((u & mask) + (X::load_off(k) & mask) > mask) return false;
            if ((X::store_base(u, k) & mask) + (X::store_off(k) & mask) > mask) return false;
        }
    return true;
}
template <class PL, int DIR, int S> __host__ __device__ constexpr int best_key(LaneMap m) {
    int best = 0, least = exchange_cost<PL, DIR, S>(m, 0);
    for (int K = 1; K < 7; ++K) {
        if (m.slots && !pad_folds<PL, DIR, S>(m, K)) continue;
        const int c = exchange_cost<PL, DIR, S>(m, K);
        if (c < least) {
            least = c;
            best = K;
        }
    }
    return best;
}
template <int K, bool PAD> __device__ __forceinline__ int exchange_slot(int base, int off) {
    if constexpr (K == 0) return base + off;
    else if constexpr (PAD) return base + (base >> K) + off + (off >> K);
    else return (base + off) ^ (((base + off) >> K) & 15);
}

// ---- stage recursion -----------------------------------------------------
// Twiddles of one plan and direction, stage after stage: entry (j - 1) P + k of
// a stage is exp(DIR 2 pi i j k / (P R)).  The lanes of a pencil hold
// consecutive k, so their loads are consecutive words (the plain table's
// stride j put whole half-warps on one bank, and its entries, kept as pairs
// to save the two moves, took five wavefronts each where these take one:
// together a fifth of the slab pass's shared-memory cycles).  tw: the table of
// a length of `every` times the plan's.
template <class PL, int DIR> __host__ __device__ constexpr int pair_tw_offset(int stage) {
    int off = 0;
    for (int s = 1; s < stage; ++s) off += (stage_radix<PL, DIR>(s) - 1) * stage_p<PL, DIR>(s);
    return off;
}
template <class PL, int DIR> __host__ __device__ constexpr int pair_tw_size() {
    return pair_tw_offset<PL, DIR>(PL::NS);
}
template <class PL, int DIR, int S = 1>
__device__ __forceinline__ void pair_tw_fill(float2* t, const float2* __restrict__ tw, int first, int step,
                                             int every = 1) {
    if constexpr (S < PL::NS) {
        constexpr int R = stage_radix<PL, DIR>(S), P = stage_p<PL, DIR>(S), STEP = PL::L / (P * R);
        for (int e = first; e < (R - 1) * P; e += step) {
            const float2 w = tw[(1 + e / P) * (e % P) * STEP * every];
            t[e] = DIR < 0 ? w : make_float2(w.x, -w.y);
        }
        pair_tw_fill<PL, DIR, S + 1>(t + (R - 1) * P, tw, first, step, every);
    }
}
// As fft_stages (fft.cuh) on NP pairs of pencils in lockstep, all of whose
// threads lie in one warp.  tw: pair_tw_fill's table.  Exchange words are two
// per position: st(slot, val) and ld(slot); the NP exchanges follow one
// another through the same words.
template <class PL, int DIR, int S, int NP, class MAP, class Ld, class St>
__device__ __forceinline__ void pair_stages(P2 (&v)[NP][PL::E], int u, const float2* tw, Ld& ld, St& st,
                                            bool half_first) {
    constexpr int L = PL::L, NT = PL::NT, E = PL::E, NS = PL::NS;
    constexpr int R = stage_radix<PL, DIR>(S), P = stage_p<PL, DIR>(S), NB = E / R;
    static_assert(E % R == 0, "radix must divide the points per thread");
    if constexpr (P > 1) {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            int k;
            if constexpr (NT % P == 0) k = u % P;
            else if constexpr (P % NT == 0) k = u + (q % (P / NT)) * NT;
            else k = (u + q * NT) % P;
#pragma unroll
            for (int j = 1; j < R; ++j) {
                const float2 w = tw[(j - 1) * P + k];
                const f32x2 c = pk(w.x, w.x), y = pk(w.y, w.y), n = pk(-w.y, -w.y);
#pragma unroll
                for (int p = 0; p < NP; ++p) v[p][q * R + j] = pmul(v[p][q * R + j], c, y, n);
            }
        }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            if constexpr (S == 0 && DIR < 0) {
                if (half_first) PDft<R, DIR>::run_half(&v[p][q * R]);
                else PDft<R, DIR>::run(&v[p][q * R]);
            } else {
                PDft<R, DIR>::run(&v[p][q * R]);
            }
        }
    if constexpr (S < NS - 1) {
        using X = ExchangePos<PL, DIR, S>;
        constexpr LaneMap LM = MAP::map();
        constexpr int K = best_key<PL, DIR, S>(LM);
        constexpr bool PAD = LM.slots != 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            __syncwarp();
#pragma unroll
            for (int k = 0; k < E; ++k) st(exchange_slot<K, PAD>(X::store_base(u, k), X::store_off(k)), v[p][k]);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < E; ++k) v[p][k] = ld(exchange_slot<K, PAD>(u, X::load_off(k)));
        }
        pair_stages<PL, DIR, S + 1, NP, MAP, Ld, St>(v, u, S == 0 ? tw : tw + (R - 1) * P, ld, st, false);
    }
}

}  // namespace dda
