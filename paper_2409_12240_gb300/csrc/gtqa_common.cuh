// Small device-side toolkit shared by the GTQA kernels: complex arithmetic,
// thread-team synchronisation, butterfly reductions and the small matrix decompositions of the
// method: one-sided Jacobi SVDs (FP32, FP64) and the FP64 SVD refined from an FP32 one.
#pragma once

#include <climits>
#include <cuda_runtime.h>
#include <stdint.h>

namespace gtqa {

// ---------------------------------------------------------------------------
// complex numbers over float or double
// ---------------------------------------------------------------------------
template <typename R>
struct __align__(sizeof(R) * 2) C {
    R x, y;
};
using cd = C<double>;
using cf = C<float>;

template <typename R> __device__ __forceinline__ C<R> cmk(R a, R b) { return C<R>{a, b}; }
template <typename R> __device__ __forceinline__ C<R> operator+(C<R> a, C<R> b) { return {a.x + b.x, a.y + b.y}; }
template <typename R> __device__ __forceinline__ C<R> operator-(C<R> a, C<R> b) { return {a.x - b.x, a.y - b.y}; }
template <typename R> __device__ __forceinline__ C<R> operator*(C<R> a, C<R> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename R> __device__ __forceinline__ C<R> operator*(R s, C<R> a) { return {s * a.x, s * a.y}; }
template <typename R> __device__ __forceinline__ C<R> conj(C<R> a) { return {a.x, -a.y}; }
template <typename R> __device__ __forceinline__ R norm2(C<R> a) { return a.x * a.x + a.y * a.y; }
// acc + a * b
template <typename R> __device__ __forceinline__ C<R> cfma(C<R> a, C<R> b, C<R> acc) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    return acc;
}
// acc + conj(a) * b
template <typename R> __device__ __forceinline__ C<R> cfmac(C<R> a, C<R> b, C<R> acc) {
    acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
    return acc;
}
// acc - a * b
template <typename R> __device__ __forceinline__ C<R> cfms(C<R> a, C<R> b, C<R> acc) {
    acc.x = fma(-a.x, b.x, fma(a.y, b.y, acc.x));
    acc.y = fma(-a.x, b.y, fma(-a.y, b.x, acc.y));
    return acc;
}
template <typename To, typename From> __device__ __forceinline__ C<To> ccast(C<From> a) {
    return C<To>{(To)a.x, (To)a.y};
}

// ---------------------------------------------------------------------------
// thread groups: G contiguous lanes inside one warp, G a power of two <= 32
// ---------------------------------------------------------------------------
template <int G>
__device__ __forceinline__ unsigned group_mask() {
    if constexpr (G >= 32) {
        return 0xffffffffu;
    } else {
        const unsigned lane = threadIdx.x & 31u;
        return ((1u << G) - 1u) << (lane & ~(unsigned)(G - 1));
    }
}

// Butterfly sum over aligned groups of G lanes.  Every lane ends with the same
// bits: at each level a lane adds a + b while its partner adds b + a.
template <int G, typename T>
__device__ __forceinline__ T group_sum(T v, unsigned mask) {
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) v += __shfl_xor_sync(mask, v, off);
    return v;
}

// Sums of NV values at once over aligned groups of G lanes.  At each butterfly level a lane hands
// the half of the values it gives up to its partner, so NV values take about NV + log2 G
// additions instead of NV log2 G (8 values over 8 lanes: 7 FP64 additions instead of 24); the
// finished sums then go to every lane by shuffles, which cost no FP64 instruction.
template <int OFF, int N, int NV, typename T>
__device__ __forceinline__ void rs_level(T (&v)[NV], unsigned mask, unsigned lane) {
    if constexpr (OFF > 0) {
        if constexpr (N == 1) {
            v[0] += __shfl_xor_sync(mask, v[0], OFF);
            rs_level<OFF / 2, 1>(v, mask, lane);
        } else {
            constexpr int H = (N + 1) / 2;
            const bool up = (lane & OFF) != 0;
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const T lo = v[i], hi = H + i < N ? v[H + i < N ? H + i : i] : (T)0;
                v[i] = (up ? hi : lo) + __shfl_xor_sync(mask, up ? lo : hi, OFF);
            }
            rs_level<OFF / 2, H>(v, mask, lane);
        }
    }
}
// lane of the group and place there that hold the sum of value i
__host__ __device__ constexpr int rs_lane(int off, int n, int i) {
    return off == 0 || n == 1 ? 0
                              : (i < (n + 1) / 2 ? rs_lane(off / 2, (n + 1) / 2, i)
                                                 : off + rs_lane(off / 2, (n + 1) / 2, i - (n + 1) / 2));
}
__host__ __device__ constexpr int rs_place(int off, int n, int i) {
    return off == 0 || n == 1 ? i
                              : (i < (n + 1) / 2 ? rs_place(off / 2, (n + 1) / 2, i)
                                                 : rs_place(off / 2, (n + 1) / 2, i - (n + 1) / 2));
}
template <int G, int I, int NV, typename T>
__device__ __forceinline__ void rs_collect(const T (&v)[NV], T (&out)[NV], unsigned mask) {
    if constexpr (I < NV) {
        out[I] = __shfl_sync(mask, v[rs_place(G / 2, NV, I)], rs_lane(G / 2, NV, I), G);
        rs_collect<G, I + 1>(v, out, mask);
    }
}
template <int G, int NV, typename T>
__device__ __forceinline__ void group_sums(T (&v)[NV], unsigned mask) {
    rs_level<G / 2, NV>(v, mask, threadIdx.x & (G - 1));
    T out[NV];
    rs_collect<G, 0>(v, out, mask);
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = out[i];
}

// Synchronisation policy for a group that lives inside one warp.
struct WarpGroup {
    unsigned mask;
    __device__ __forceinline__ void sync() const { __syncwarp(mask); }
    __device__ __forceinline__ bool any(int p) const { return __any_sync(mask, p) != 0; }
    __device__ __forceinline__ int max_int(int v) const { return __reduce_max_sync(mask, v); }
    __device__ __forceinline__ unsigned or_bits(unsigned v) const { return __reduce_or_sync(mask, v); }
};

// Synchronisation policy for a group that is the whole thread block.
struct BlockGroup {
    int* flag;  // one int of shared memory
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    __device__ __forceinline__ bool any(int p) const {
        __syncthreads();
        if (threadIdx.x == 0) *flag = 0;
        __syncthreads();
        if (p) atomicOr(flag, 1);
        __syncthreads();
        return *flag != 0;
    }
    __device__ __forceinline__ int max_int(int v) const {
        __syncthreads();
        if (threadIdx.x == 0) *flag = INT_MIN;
        __syncthreads();
        atomicMax(flag, v);
        __syncthreads();
        return *flag;
    }
    __device__ __forceinline__ unsigned or_bits(unsigned v) const {
        __syncthreads();
        if (threadIdx.x == 0) *flag = 0;
        __syncthreads();
        if (v) atomicOr(reinterpret_cast<unsigned*>(flag), v);
        __syncthreads();
        return *reinterpret_cast<volatile unsigned*>(flag);
    }
};

// ---------------------------------------------------------------------------
// Reciprocal and (reciprocal) square root without the FP64 divide/sqrt sequences,
// which cost ~10-15 FP64 pipe instructions each on this part.  A hardware seed
// (PTX rcp.approx.ftz.f64 / rsqrt.approx.ftz.f64, ~2^-22 relative error) is refined by one
// third-order step (error e -> O(e^3) ~ 2^-63, i.e. FP64 rounding): 3 and 5 FP64 instructions,
// against 4 and 8 for two Newton steps.
// Float versions use the single-precision hardware approximations directly.
// Inputs must be finite and positive (callers guard zero).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double nr_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);   // r (1 + e + e^2)
}
// one refinement step only: relative error ~2^-44, for results that are rounded to FP32
__device__ __forceinline__ double nr_rcp1(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ double nr_rsqrt(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);   // y (1 + e/2 + 3 e^2/8)
}
__device__ __forceinline__ double nr_sqrt(double x) {
    if (!(x > 0.0)) return 0.0;
    const double y = nr_rsqrt(x);
    const double s = x * y;
    return fma(0.5 * y, fma(-s, s, x), s);   // one correction of s = sqrt(x)
}
__device__ __forceinline__ float nr_rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ float nr_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ float nr_sqrt(float x) { return x > 0.f ? sqrtf(x) : 0.f; }

// ---------------------------------------------------------------------------
// Batched one-sided (Hestenes) Jacobi SVD of an N x N complex matrix.
//
// A and V are column-major in shared memory (element (row r, col c) at c*N + r).
// The group has N*N/2 threads: thread g works on pair k = g / N at row r = g % N,
// so the N lanes of a pair are contiguous and reduce with shuffles.  Columns are
// paired by the round-robin (circle) ordering, N/2 disjoint pairs per step and
// N-1 steps per sweep.  For a pair (p, q) with alpha = |a_p|^2, beta = |a_q|^2,
// gamma = a_p^H a_q, the 2x2 unitary J = [[c, s e],[-s conj(e), c]] (e = gamma/|gamma|,
// t = tan(theta) the smaller root of t^2 + 2 zeta t - 1 = 0, zeta = (beta-alpha)/(2|gamma|))
// makes the rotated columns orthogonal.  Sweeps stop when no pair has
// |gamma| > tol * sqrt(alpha beta).  On exit A holds U*S (columns unsorted) and
// V the accumulated right rotations: A_in = (A_out) V^H.
// ---------------------------------------------------------------------------
// Zeroes the entries of an N x N complex matrix (column-major, shared) that lie more than 2^100
// (about 1e30) below its largest entry.  Every value kept by the method's cut-offs (singular
// values above 1e-14 s_0, message eigenvalues above 1e-13 w_max) is far above that, while such
// rounding-level columns would keep one-sided Jacobi rotating pairs whose angle underflows
// (a column of norm ~1e-44 next to one of norm ~1 in the early anneal).  The test compares the
// exponent bits of the entries, on the integer pipe.  The group has N^2/2 lanes.
__device__ __forceinline__ int exp_bits(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff); }
template <int N, typename Group>
__device__ void prune_noise(C<double>* A, int g, const Group& grp) {
    constexpr int NN = N * N, L = NN / 2;
    int e = 0;
#pragma unroll
    for (int j = 0; j < NN / L; ++j) {
        const C<double> a = A[g + j * L];
        e = max(e, max(exp_bits(a.x), exp_bits(a.y)));
    }
    const int emax = grp.max_int(e);
#pragma unroll
    for (int j = 0; j < NN / L; ++j) {
        const C<double> a = A[g + j * L];
        if (max(exp_bits(a.x), exp_bits(a.y)) < emax - 100) A[g + j * L] = C<double>{0.0, 0.0};
    }
    grp.sync();
}

__device__ __forceinline__ void round_robin_pair(int N, int step, int k, int& p, int& q) {
    if (k == 0) {
        p = step;
        q = N - 1;
    } else {
        p = (step + k) % (N - 1);
        q = (step - k + (N - 1)) % (N - 1);
    }
    if (p > q) { int t = p; p = q; q = t; }
}

// Options: WITHV = false skips the V updates (only the singular values are wanted).
// F32ANGLE (R = double): the rotation angle t is solved in FP32 from the FP64 zeta, and c,
// s and the phase e are then formed in FP64 from that t, so every rotation is unitary to
// FP64 rounding and the FP64 orthogonality test decides convergence; only the size of
// each step is FP32-accurate.  quad_tol > 0: a sweep whose examined pairs all have
// |gamma| <= quad_tol sqrt(alpha beta) is the last one: with quadratic convergence the
// next sweep would find |gamma| ~ quad_tol^2 sqrt(alpha beta) <= tol sqrt(alpha beta) (for
// quad_tol^2 <= tol), so the confirming sweep is skipped.
template <int N, typename R, typename Group, bool WITHV = true, bool F32ANGLE = false>
__device__ int jacobi_svd(C<R>* A, C<R>* V, int g, const Group& grp, unsigned pair_mask,
                          R tol, int max_sweeps, bool init_v, int* nrot = nullptr, R quad_tol = (R)0) {
    const int k = g / N;
    const int r = g % N;
    if (WITHV && init_v) {
        V[(2 * k) * N + r] = C<R>{(R)((2 * k) == r), (R)0};
        V[(2 * k + 1) * N + r] = C<R>{(R)((2 * k + 1) == r), (R)0};
    }
    grp.sync();
    const R tol2 = tol * tol, quad2 = quad_tol * quad_tol;
    // a pair whose |gamma|^2 lies near the bottom of the range is orthogonal in absolute terms
    // (the matrices here are normalised); taking it as converged also keeps the reciprocal
    // square root away from subnormal inputs
    const R gmin = sizeof(R) == 8 ? (R)1e-290 : (R)1e-36;
    const bool quad = quad_tol > (R)0;
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        int rotated = 0, big = 0;
        for (int step = 0; step < N - 1; ++step) {
            int p, q;
            round_robin_pair(N, step, k, p, q);
            C<R> ap = A[p * N + r], aq = A[q * N + r];
            R alpha = norm2(ap), beta = norm2(aq);
            C<R> gam = cfmac(ap, aq, C<R>{(R)0, (R)0});
            alpha = group_sum<N>(alpha, pair_mask);
            beta = group_sum<N>(beta, pair_mask);
            gam.x = group_sum<N>(gam.x, pair_mask);
            gam.y = group_sum<N>(gam.y, pair_mask);
            const R g2 = gam.x * gam.x + gam.y * gam.y;
            const R ab = alpha * beta;
            if (g2 > gmin && g2 > tol2 * ab) {
                if (g2 > quad2 * ab) big = 1;
                const R rg = nr_rsqrt(g2);                      // 1 / |gamma|
                const R zeta = (beta - alpha) * ((R)0.5 * rg);
                R t;
                if constexpr (F32ANGLE) {
                    // t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)) in FP32; for huge zeta (beyond the FP32
                    // range when a column is tiny) t = 1/(2 zeta) in FP64, so the rotation does not vanish
                    const R az = fabs(zeta);
                    if (az < (R)1e18) {
                        const float azf = (float)az;
                        const float tf = __frcp_rn(azf + sqrtf(fmaf(azf, azf, 1.f)));
                        t = (R)(zeta >= (R)0 ? tf : -tf);
                    } else {
                        t = (zeta >= (R)0 ? (R)0.5 : (R)-0.5) * nr_rcp(az);
                    }
                } else {
                    const R az = fabs(zeta);
                    // t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)), the smaller root; 1/(2 zeta) for huge zeta
                    t = (zeta >= (R)0 ? (R)1 : (R)-1) *
                        (az < (R)1e15 ? nr_rcp(az + nr_sqrt((R)1 + az * az)) : (R)0.5 * nr_rcp(az));
                }
                const R c = nr_rsqrt((R)1 + t * t);
                const R s = c * t;
                const C<R> e = C<R>{gam.x * rg, gam.y * rg};
                const C<R> se = s * e;
                const C<R> sec = conj(se);
                A[p * N + r] = c * ap - sec * aq;
                A[q * N + r] = se * ap + c * aq;
                if constexpr (WITHV) {
                    const C<R> vp = V[p * N + r], vq = V[q * N + r];
                    V[p * N + r] = c * vp - sec * vq;
                    V[q * N + r] = se * vp + c * vq;
                }
                rotated = 1;
                if (nrot && r == 0) ++*nrot;
            }
            grp.sync();
        }
        if (!grp.any(quad ? big : rotated)) {
            ++sweep;
            break;
        }
    }
    return sweep;   // sweeps run, including the final one (without rotations unless quad_tol stopped it)
}

// hardware approximations (about 2^-22), for rotation angles
__device__ __forceinline__ float fast_sqrt(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// The right singular vectors of an FP32 N x N matrix by one-sided Jacobi (the stopping rule of
// jacobi_svd with tol 1e-6 and quad_tol 1e-3), for a group of N^2 / 2 <= 32 lanes: lane (k, r)
// keeps row r of the two columns of pair k, and of V, in registers.  The circle ordering
// moves one column of every pair to each neighbouring pair per step, by shuffles, so a step has
// no shared-memory round trip and no index arithmetic: it is the latency of three shuffle
// levels, the angle (one square root, one reciprocal, one reciprocal square root) and the move
// (460 cycles per step of N = 8, against about 700 through shared memory).  keep < N: pairs without
// a column among the keep largest (norms within a factor 4 of the keep-th count) do not ask for
// another sweep, and a kept column with a smaller one is judged by the kept column's norm, as in
// refined_svd; that saves 0.6 to 1 of 4.6 to 5.3 sweeps of the gates.  OUT: A ends as U S.
template <int N, bool OUT = false>
__device__ int jacobi_v32(C<float>* A, C<float>* V, int g, unsigned gmask, unsigned pair_mask, int keep) {
    using CF = C<float>;
    constexpr int LN = N * N / 2, LAST = N / 2 - 1;
    static_assert(LN <= 32, "the group lives in one warp");
    const int k = g / N, r = g % N;
    CF a = A[k * N + r], b = A[(N - 1 - k) * N + r];
    CF va = CF{k == r ? 1.f : 0.f, 0.f}, vb = CF{N - 1 - k == r ? 1.f : 0.f, 0.f};
    int sweep = 0;
    for (; sweep < 40; ++sweep) {
        int big = 0;
        float thr = 0.f;   // a quarter of the keep-th largest squared norm
        for (int step = 0; step < N - 1; ++step) {
            float s[4] = {norm2(a), norm2(b), fmaf(a.x, b.x, a.y * b.y), fmaf(a.x, b.y, -a.y * b.x)};
#pragma unroll
            for (int o = N / 2; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) s[i] += __shfl_xor_sync(pair_mask, s[i], o);
            const float g2 = fmaf(s[2], s[2], s[3] * s[3]), ab = s[0] * s[1];
            const bool rot = g2 > 1e-36f && g2 > 1e-12f * ab;
            if (N > 2 && step == 0 && keep < N) {
                int ca = 0, cb = 0;   // columns at least as long as this pair's two
                for (int j = 0; j < N / 2; ++j) {
                    const float x = __shfl_sync(gmask, s[0], j * N, LN), y = __shfl_sync(gmask, s[1], j * N, LN);
                    ca += (x >= s[0]) + (y >= s[0]);
                    cb += (x >= s[1]) + (y >= s[1]);
                }
                const float x = fmaxf(ca >= keep ? s[0] : 0.f, cb >= keep ? s[1] : 0.f);
                thr = 0.25f * __int_as_float(__reduce_max_sync(gmask, __float_as_int(x)));
            }
            const float mx = fmaxf(s[0], s[1]), lim = fminf(s[0], s[1]) >= thr ? ab : mx * mx;
            if (rot && mx >= thr && g2 > 1e-6f * lim) big = 1;
            const float d = s[1] - s[0];
            const float tn = 2.f * fast_rcp(fabsf(d) + fast_sqrt(fmaf(d, d, 4.f * g2)));
            const float tau = rot ? (d >= 0.f ? tn : -tn) : 0.f;
            const float c = rot ? rsqrtf(fmaf(tau * tau, g2, 1.f)) : 1.f;
            const CF se = CF{c * tau * s[2], c * tau * s[3]};
            const CF na = CF{fmaf(-se.x, b.x, fmaf(-se.y, b.y, c * a.x)), fmaf(-se.x, b.y, fmaf(se.y, b.x, c * a.y))};
            const CF nb = CF{fmaf(se.x, a.x, fmaf(-se.y, a.y, c * b.x)), fmaf(se.x, a.y, fmaf(se.y, a.x, c * b.y))};
            const CF ma = CF{fmaf(-se.x, vb.x, fmaf(-se.y, vb.y, c * va.x)), fmaf(-se.x, vb.y, fmaf(se.y, vb.x, c * va.y))};
            const CF mb = CF{fmaf(se.x, va.x, fmaf(-se.y, va.y, c * vb.x)), fmaf(se.x, va.y, fmaf(se.y, va.x, c * vb.y))};
            if constexpr (N > 2) {
                // first column: from pair k + 1 (the last pair: its own second one); second column:
                // from pair k - 1 (pair 1: the first one of pair 0; pair 0 keeps its own)
                auto first = [&](float x, float y) {
                    const float t = __shfl_down_sync(gmask, x, N, LN);
                    return k == LAST ? y : t;
                };
                auto second = [&](float x, float y) {
                    const float t = __shfl_up_sync(gmask, k == 0 ? x : y, N, LN);
                    return k == 0 ? y : t;
                };
                a = CF{first(na.x, nb.x), first(na.y, nb.y)};
                b = CF{second(na.x, nb.x), second(na.y, nb.y)};
                va = CF{first(ma.x, mb.x), first(ma.y, mb.y)};
                vb = CF{second(ma.x, mb.x), second(ma.y, mb.y)};
            } else {
                a = na;
                b = nb;
                va = ma;
                vb = mb;
            }
        }
        if (!__any_sync(gmask, big)) {
            ++sweep;
            break;
        }
    }
    // after a whole sweep every column is back at its pair
    V[k * N + r] = va;
    V[(N - 1 - k) * N + r] = vb;
    if constexpr (OUT) {
        A[k * N + r] = a;
        A[(N - 1 - k) * N + r] = b;
    }
    return sweep;
}

// The same for a group of several warps (N = 16, 32): the columns go to the neighbouring pairs
// through shared memory, in two buffers used in turn, so that a step has one barrier.  A, V: N^2
// entries each; buf: 2 N^2 entries; nrm: 2 N floats.  V32 ends in V.
template <int N, bool OUT, typename Group>
__device__ int jacobi_v32_team(C<float>* A, C<float>* V, C<float>* buf, float* nrm, int g, const Group& grp,
                               unsigned pair_mask, int keep) {
    using CF = C<float>;
    constexpr int NN = N * N, LAST = N / 2 - 1;
    const int k = g / N, r = g % N;
    // the slots (2 k: first column of pair k, 2 k + 1: second) that this pair's columns move to
    const int da = (k == 0 ? 3 : 2 * (k - 1)) * N + r, db = (k == 0 ? 1 : (k == LAST ? 2 * LAST : 2 * (k + 1) + 1)) * N + r;
    const int sa = 2 * k * N + r, sb = sa + N;
    CF a = A[k * N + r], b = A[(N - 1 - k) * N + r];
    CF va = CF{k == r ? 1.f : 0.f, 0.f}, vb = CF{N - 1 - k == r ? 1.f : 0.f, 0.f};
    int sweep = 0, par = 0;
    for (; sweep < 40; ++sweep) {
        int big = 0;
        float thr = 0.f;
        for (int step = 0; step < N - 1; ++step) {
            float s[4] = {norm2(a), norm2(b), fmaf(a.x, b.x, a.y * b.y), fmaf(a.x, b.y, -a.y * b.x)};
            group_sums<N>(s, pair_mask);
            const float g2 = fmaf(s[2], s[2], s[3] * s[3]), ab = s[0] * s[1];
            const bool rot = g2 > 1e-36f && g2 > 1e-12f * ab;
            if (step == 0 && keep < N) {
                if (r == 0) {
                    nrm[2 * k] = s[0];
                    nrm[2 * k + 1] = s[1];
                }
                grp.sync();
                // a quarter of the keep-th largest squared norm
                if (g < N) {
                    const float x = nrm[g];
                    int c = 0;
                    for (int i = 0; i < N; ++i) c += nrm[i] >= x;
                    nrm[N + g] = c >= keep ? 0.25f * x : 0.f;
                }
                grp.sync();
                for (int j = 0; j < N; ++j) thr = fmaxf(thr, nrm[N + j]);
                grp.sync();
            }
            const float mx = fmaxf(s[0], s[1]), lim = fminf(s[0], s[1]) >= thr ? ab : mx * mx;
            if (rot && mx >= thr && g2 > 1e-6f * lim) big = 1;
            const float d = s[1] - s[0];
            const float tn = 2.f * fast_rcp(fabsf(d) + fast_sqrt(fmaf(d, d, 4.f * g2)));
            const float tau = rot ? (d >= 0.f ? tn : -tn) : 0.f;
            const float c = rot ? rsqrtf(fmaf(tau * tau, g2, 1.f)) : 1.f;
            const CF se = CF{c * tau * s[2], c * tau * s[3]};
            CF* bA = par ? buf : A;
            CF* bV = par ? buf + NN : V;
            par ^= 1;
            if (step == 0 && sweep == 0) grp.sync();   // every lane has its columns of A
            bA[da] = CF{fmaf(-se.x, b.x, fmaf(-se.y, b.y, c * a.x)), fmaf(-se.x, b.y, fmaf(se.y, b.x, c * a.y))};
            bA[db] = CF{fmaf(se.x, a.x, fmaf(-se.y, a.y, c * b.x)), fmaf(se.x, a.y, fmaf(se.y, a.x, c * b.y))};
            bV[da] = CF{fmaf(-se.x, vb.x, fmaf(-se.y, vb.y, c * va.x)), fmaf(-se.x, vb.y, fmaf(se.y, vb.x, c * va.y))};
            bV[db] = CF{fmaf(se.x, va.x, fmaf(-se.y, va.y, c * vb.x)), fmaf(se.x, va.y, fmaf(se.y, va.x, c * vb.y))};
            grp.sync();
            a = bA[sa];
            b = bA[sb];
            va = bV[sa];
            vb = bV[sb];
        }
        if (!grp.any(big)) {
            ++sweep;
            break;
        }
    }
    grp.sync();
    V[k * N + r] = va;
    V[(N - 1 - k) * N + r] = vb;
    if constexpr (OUT) {
        A[k * N + r] = a;
        A[(N - 1 - k) * N + r] = b;
    }
    return sweep;
}

// True if x (an updated squared norm) is negative, zero or below about half of ref, from the
// raw bits only.
__device__ __forceinline__ bool norm_collapsed(double x, double ref) {
    const long long b = __double_as_longlong(x);
    return b <= 0 || (int)((b >> 52) & 0x7ff) + 1 < exp_bits(ref);
}

// FP64 polish of a one-sided Jacobi SVD (same layout, pairing and rotations as
// jacobi_svd<N, double>) for columns that are already nearly orthogonal, as
// refined_svd leaves those that its passes do not close.  Fewer FP64 instructions per step:
//  * the squared column norms are kept in nrm[N] (shared) and, in steps whose rotations are all
//    small, updated as alpha' = alpha - tau |gamma|^2 and beta' = beta + tau |gamma|^2 (the two
//    eigenvalues of the pair's 2x2 Gram matrix) instead of two reductions per step; after a
//    large rotation, or where the update would remove more than half of a norm (it then
//    cancels), they are recomputed;
//  * the rotation is parametrised by tau = t / |gamma| = 2 sign(D) / (|D| + sqrt(D^2 + 4|gamma|^2)),
//    D = beta - alpha, solved in FP32 on values scaled by an approximate 1/(alpha + beta);
//    then t^2 = tau^2 |gamma|^2, c = 1/sqrt(1 + t^2) and s e = c tau gamma are formed in FP64,
//    so c^2 + |s e|^2 = 1 to FP64 rounding whatever the error of tau, and the FP64
//    orthogonality test alone decides convergence;
//  * c = 1 - t^2/2 + 3t^4/8 when every pair of the group has t^2 < 1e-6 (the dropped terms are
//    below 3.2e-19).
// The quadratic stop of jacobi_svd applies (quad_tol).
// keep_rank < N (the caller keeps at most keep_rank singular triplets, as in the truncation of
// App. D): only pairs that touch a column among the keep_rank largest (with a margin: norms
// within a factor 4 of the keep_rank-th largest at entry count) decide the quadratic stop, and
// a pair of such a column p with a smaller one q is judged by |gamma| against alpha_p (the
// size of the rotation of the kept column) rather than sqrt(alpha_p beta_q).  The kept
// columns then converge as with keep_rank = N, while rotations among discarded columns, which
// leave the kept subspace unchanged, no longer force a confirming sweep.
// The first sweep runs first_steps (all by default); a later sweep runs only the steps of the
// round-robin schedule in which the previous sweep made a rotation above quad_tol.  A pair
// whose rotation in a sweep stayed below quad_tol is orthogonal after it to about quad_tol
// times the largest rotation of that sweep (the rotations of its columns with the others
// reintroduce only products of their sizes), which is the accuracy of the quadratic stop, so
// those steps need no second pass.
// Returns the sweeps run (partial ones included); *nsteps (if given, group lane 0) counts the
// steps run, of N / 2 pairs each.
template <int N, typename Group>
__device__ int jacobi_polish(C<double>* A, C<double>* V, double* nrm, int g, const Group& grp, unsigned pair_mask,
                             double tol, double quad_tol, int max_sweeps, int* nrot, int keep_rank = N,
                             unsigned* relmask = nullptr, int* nsteps = nullptr, unsigned first_steps = ~0u) {
    using CD = C<double>;
    const int k = g / N;
    const int r = g % N;
    {
        const double n0 = group_sum<N>(norm2(A[(2 * k) * N + r]), pair_mask);
        const double n1 = group_sum<N>(norm2(A[(2 * k + 1) * N + r]), pair_mask);
        if (r == 0) {
            nrm[2 * k] = n0;
            nrm[2 * k + 1] = n1;
        }
    }
    grp.sync();
    const bool partial = keep_rank < N && relmask != nullptr;
    if (partial) {
        if (g == 0) *relmask = 0u;
        grp.sync();
        if (g < N) {
            // the keep_rank-th largest norm, then every column within a factor 4 of it
            const double x = nrm[g];
            int above = 0;
            for (int j = 0; j < N; ++j) above += (nrm[j] > x) || (nrm[j] == x && j < g);
            if (above == keep_rank - 1) {
                const double thr = 0.25 * x;
                unsigned mask = 0u;
                for (int j = 0; j < N; ++j) mask |= (nrm[j] >= thr) ? (1u << j) : 0u;
                *relmask = mask;
            }
        }
        grp.sync();
    }
    const unsigned rel = partial ? *relmask : 0xffffffffu;
    const double tol2 = tol * tol, quad2 = quad_tol * quad_tol;
    static_assert(N - 1 < 32, "one bit per step");
    unsigned steps = ((1u << (N - 1)) - 1u) & first_steps;   // steps this sweep runs
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        unsigned bigsteps = 0u;   // this lane's steps with a rotation above quad_tol
        for (int step = 0; step < N - 1; ++step) {
            if (!((steps >> step) & 1u)) continue;   // the same for the whole group
            int bstep = 0;   // this lane's pair rotated by more than quad_tol
            if (nsteps && g == 0) ++*nsteps;
            int p, q;
            round_robin_pair(N, step, k, p, q);
            const CD ap = A[p * N + r], aq = A[q * N + r];
            const double alpha = nrm[p], beta = nrm[q];
            CD gam = cfmac(ap, aq, CD{0.0, 0.0});
            gam.x = group_sum<N>(gam.x, pair_mask);
            gam.y = group_sum<N>(gam.y, pair_mask);
            const double g2 = gam.x * gam.x + gam.y * gam.y;
            const double ab = alpha * beta;
            const bool rot = g2 > 1e-290 && g2 > tol2 * ab;   // as in jacobi_svd
            double tau = 0.0, t2 = 0.0;
            if (rot) {
                const bool rp = (rel >> p) & 1u, rq = (rel >> q) & 1u;
                if (rp && rq) {
                    if (g2 > quad2 * ab) bstep = 1;
                } else if (rp || rq) {
                    const double mx = alpha > beta ? alpha : beta;
                    if (g2 > quad2 * mx * mx) bstep = 1;
                }
                const double d = beta - alpha;
                double rsc;
                asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(rsc) : "d"(alpha + beta));
                const float dn = (float)(d * rsc), gn = (float)(g2 * rsc * rsc);
                const float tn = 2.f * __frcp_rn(fabsf(dn) + sqrtf(fmaf(dn, dn, 4.f * gn)));
                tau = (double)(dn >= 0.f ? tn : -tn) * rsc;
                t2 = tau * tau * g2;
            }
            const bool series = !grp.any(rot && !(t2 < 1e-6));
            if (rot) {
                const double c = series ? fma(t2, fma(0.375, t2, -0.5), 1.0) : nr_rsqrt(1.0 + t2);
                const double ct = c * tau;
                const CD se = CD{ct * gam.x, ct * gam.y};
                const CD sec = conj(se);
                A[p * N + r] = c * ap - sec * aq;
                A[q * N + r] = se * ap + c * aq;
                const CD vp = V[p * N + r], vq = V[q * N + r];
                V[p * N + r] = c * vp - sec * vq;
                V[q * N + r] = se * vp + c * vq;
                if (r == 0 && nrot) ++*nrot;
            }
            // the updated norms; the smaller one loses |m|, and where that cancels (a column nearly
            // parallel to a larger one) the update loses its precision and can turn negative, so
            // both are then recomputed from the columns, as after a large rotation.  The test
            // reads the sign and exponent bits (integer pipe): a drop below half or a sign change
            const double m = tau * g2;   // 0 without a rotation
            const double np_ = alpha - m, nq_ = beta + m;
            const bool exact = !series || (rot && (norm_collapsed(np_, alpha) || norm_collapsed(nq_, beta)));
            if (!exact) {
                if (rot && r == 0) {
                    nrm[p] = np_;
                    nrm[q] = nq_;
                }
            } else {
                // a large rotation: the update alpha - tau |gamma|^2 can cancel, so the two
                // norms are recomputed from the rotated columns
                const double np = group_sum<N>(norm2(A[p * N + r]), pair_mask);
                const double nq = group_sum<N>(norm2(A[q * N + r]), pair_mask);
                if (r == 0) {
                    nrm[p] = np;
                    nrm[q] = nq;
                }
            }
            if (bstep) bigsteps |= 1u << step;
            grp.sync();
        }
        steps = grp.or_bits(bigsteps);
        if (!steps) {
            ++sweep;
            break;
        }
    }
    return sweep;
}

// ---------------------------------------------------------------------------
// FP64 SVD of an N x N complex matrix (column-major, shared memory) from an FP32 one.
//
// What bounds it: the FP64 pipe (one warp instruction per 64 cycles and sub-partition, whatever
// its active lanes).  An FP64 Jacobi sweep costs N - 1 dependent steps of about 57 FP64
// instructions per warp (N = 8: 400), and a decomposition needs 6 to 11 of them; a pass of the
// refinement below costs two or three N^3 products (N = 8: 130 to 200), all lanes busy and no
// chain of steps, and one or two passes suffice:
//   1. one-sided Jacobi on an FP32 copy (scaled by the exponent of its largest entry) gives V32;
//   2. V = V32 is made unitary: V <- V (I - E/2), E = V^H V - I in compensated FP32, the
//      correction's product in FP32 (|E| ~ 1e-6, so its rounding lies near 1e-13); F64: once more
//      with an FP64 Gram product, which leaves rounding level;
//   3. W = A V in FP64;
//   4. passes: the Gram matrix of W in FP64, every pair's rotation parameter (as in
//      jacobi_polish: K_pq = tau gamma_pq) at once, and W <- W (I + K + K^2/2), V likewise, for
//      all pairs with |K_pq| <= 1e-4.  K is antihermitian, so the factor is unitary up to
//      ||K||^4/4 and the FP32 rounding of K^2: V^H V - I stays below 4e-15 (N = 8), 1e-14 (16) and 4e-14 (32)
//      on clustered and graded spectra, whose K are the largest, and near 1e-15 elsewhere.  (Taking V's defect out in the
//      next pass leaves 1e-15 everywhere for 1.5 % of an FP64 anneal: not done, FP64 Jacobi sweeps
//      accumulate 3e-15 to 8e-15.)  The off-diagonals shrink to products of their sizes.  Without F64 the
//      corrections are formed in FP32 where every kept column moves by less than 1e-3 of its length
//      (12 FP64 instructions per warp instead of 64).  A pair is open, and asks for another pass, while
//      its cosine is above `stop` or, unless the cosine is below tol, its |K| above 1e-8 (1e-4 without
//      F64): columns of nearly the same length take a large rotation at a small cosine.  With F64 the
//      products of the columns that do not count enter K and the end too, where they are long and
//      not orthogonal to each other.
//      A pair with a larger K (nearly equal or not yet resolved columns) is rotated by
//      FP64 Jacobi steps (only the steps of the schedule that hold such a pair) or, for N >= 16
//      with many of them, by FP32 Jacobi on those and all shorter columns of W, rescaled,
//      which resolves the columns that lay below the FP32 resolution of the first stage.
//   A decomposition that is still open after MAXP passes goes to jacobi_polish.
// Cores of whole anneals (n = 300, chi = 4): 1.3 passes on average in the mixed mode, 2.1 with
// F64; chi = 8 2.0 and 2.8, chi = 16 (F64) 1.9.  Orthogonality of the kept columns after it: 2e-10
// (stop 1e-5) and 1e-15 (F64).  Kept triplets with a relative gap d to the first discarded one: 1e-16 / d (F64).
// ---------------------------------------------------------------------------
// The pair of columns of lane g: the N (N - 1) / 2 pairs in the order of the Jacobi schedule
// (lane g: pair g % (N / 2) of step g / (N / 2)); false for the lanes that are left over.
template <int N>
__device__ __forceinline__ bool lane_pair(int g, int& step, int& p, int& q) {
    step = g / (N / 2);
    p = 0;
    q = N > 1 ? 1 : 0;
    if (step >= N - 1) return false;
    round_robin_pair(N, step, g % (N / 2), p, q);
    return true;
}
// Squared column norms into nrm[N] (N / 2 lanes per column, two rows each); no synchronisation.
template <int N>
__device__ __forceinline__ void column_norms(const C<double>* A, double* nrm, int g) {
    constexpr int H = N / 2;
    const int c = g / H, r = g % H;
    double s = norm2(A[c * N + r]) + norm2(A[c * N + r + H]);
    s = group_sum<H>(s, group_mask<(H < 32 ? H : 32)>());
    if (r == 0) nrm[c] = s;
}
// Column norms into nrm, and a_p^H a_q of the lane's pair.  The rows start at the lane's own, so
// that the lanes of a warp read different banks.
template <int N, typename Group>
__device__ __forceinline__ C<double> gram(const C<double>* A, double* nrm, int g, const Group& grp, bool has, int p,
                                          int q) {
    column_norms<N>(A, nrm, g);
    C<double> gam = C<double>{0.0, 0.0};
    if (has)
        for (int i = 0; i < N; ++i) {
            const int r = (i + g) & (N - 1);
            gam = cfmac(A[p * N + r], A[q * N + r], gam);
        }
    grp.sync();
    return gam;
}
// acc + a b with the rounding errors of the product and of the sum collected in err (Dekker / Knuth
// two-product and two-sum; the result acc + err has about twice the FP32 precision)
__device__ __forceinline__ void dot2(float a, float b, float& acc, float& err) {
    const float p = __fmul_rn(a, b), e = fmaf(a, b, -p);   // (intrinsics: not to be contracted)
    const float t = __fadd_rn(acc, p), z = __fsub_rn(t, acc);
    err += e + (__fsub_rn(acc, __fsub_rn(t, z)) + __fsub_rn(p, z));
    acc = t;
}
// -(V^H V - I) / 2 of an FP32 matrix into L.  The entries are differences of about 1e-6 and are
// needed to 1e-12: twice the FP32 precision in FP32 instructions (about 40 per complex product,
// against 4 FP64 ones that take 64 cycles each).
template <int N, typename Group>
__device__ __forceinline__ void half_defect32(const C<float>* V, C<float>* L, int g, const Group& grp, bool has, int p,
                                              int q) {
    if (has) {
        float x = 0.f, xe = 0.f, y = 0.f, ye = 0.f;
        for (int i = 0; i < N; ++i) {
            const int r = (i + g) & (N - 1);
            const C<float> a = V[p * N + r], b = V[q * N + r];
            dot2(a.x, b.x, x, xe);
            dot2(a.x, b.y, y, ye);
            dot2(a.y, b.y, x, xe);
            dot2(-a.y, b.x, y, ye);
        }
        const C<float> e = C<float>{-0.5f * (x + xe), -0.5f * (y + ye)};
        L[q * N + p] = e;
        L[p * N + q] = conj(e);
    }
    if (g < N) {
        float x = -1.f, xe = 0.f;
        for (int r = 0; r < N; ++r) {
            const C<float> a = V[g * N + r];
            dot2(a.x, a.x, x, xe);
            dot2(a.y, a.y, x, xe);
        }
        L[g * N + g] = C<float>{-0.5f * (x + xe), 0.f};
    }
    grp.sync();
}
// X <- X + X32 L with the product in FP32, X32 <- X rounded first.
template <int N, typename Group>
__device__ __forceinline__ void correct32(C<double>* X, C<float>* X32, const C<float>* L, int g, const Group& grp) {
    constexpr int LN = N * N / 2;
#pragma unroll
    for (int j = 0; j < 2; ++j) X32[g + j * LN] = ccast<float>(X[g + j * LN]);
    grp.sync();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int t = g + j * LN, q = t / N, r = t % N;
        C<float> acc = C<float>{0.f, 0.f};
        for (int p = 0; p < N; ++p) acc = cfma(X32[p * N + r], L[q * N + p], acc);
        X[t] = X[t] + ccast<double>(acc);
    }
    grp.sync();
}
// V <- V + V32 L with the product in FP32, and V32 <- V rounded.
template <int N, typename Group>
__device__ __forceinline__ void add_product32(C<double>* V, C<float>* V32, const C<float>* L, int g, const Group& grp) {
    constexpr int LN = N * N / 2;
    C<float> acc[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int t = g + j * LN, q = t / N, r = t % N;
        acc[j] = C<float>{0.f, 0.f};
        for (int p = 0; p < N; ++p) acc[j] = cfma(V32[p * N + r], L[q * N + p], acc[j]);
    }
    grp.sync();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int t = g + j * LN;
        const C<double> v = V[t] + ccast<double>(acc[j]);
        V[t] = v;
        V32[t] = ccast<float>(v);
    }
    grp.sync();
}
// X <- X B (ADD: X + X B) in FP64, in place.
template <int N, bool ADD, typename Group>
__device__ __forceinline__ void mul64(C<double>* X, const C<double>* B, int g, const Group& grp) {
    constexpr int LN = N * N / 2;
    C<double> acc[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int t = g + j * LN, q = t / N, r = t % N;
        acc[j] = ADD ? X[t] : C<double>{0.0, 0.0};
        for (int p = 0; p < N; ++p) acc[j] = cfma(X[p * N + r], B[q * N + p], acc[j]);
    }
    grp.sync();
#pragma unroll
    for (int j = 0; j < 2; ++j) X[g + j * LN] = acc[j];
    grp.sync();
}
// 2^-e for the exponent field `bits` of a normal double; 0 for a zero, subnormal or non-finite one
__device__ __forceinline__ double inv_exp2(int bits) {
    return bits > 0 && bits < 2046 ? __longlong_as_double((long long)(2046 - bits) << 52) : 0.0;
}

// squared norms at or below this count as zero (their reciprocal roots leave the range)
template <typename R> __host__ __device__ constexpr R tiny_norm2() { return 1e-300; }
template <> __host__ __device__ constexpr float tiny_norm2<float>() { return 0.f; }
// whether a non-negative value is not zero, from its bits (no FP64 compare)
__device__ __forceinline__ bool nonzero(double x) { return __double_as_longlong(x) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.f; }

struct SvdCount {       // work of one decomposition
    int passes = 0;     // refinement passes (and sweeps of a closing jacobi_polish)
    int sweeps32 = 0;   // FP32 sweeps
    int pairs = 0;      // pairs examined in FP64: N (N - 1) / 2 per pass, N / 2 per Jacobi step
    int rot = 0;        // FP64 Jacobi rotations of this lane's pairs
};

// V32's Jacobi run on the FP32 copy in A32, and V (FP64) from it, unitary to ~1e-12 (F64: to
// rounding).  V32 holds V rounded afterwards.
template <int N, bool F64, typename Group>
__device__ int svd32_unitary(C<double>* V, C<float>* A32, C<float>* V32, double* nrm, int g, const Group& grp,
                             unsigned pair_mask, int keep) {
    constexpr int LN = N * N / 2;
    int step, p, q;
    const bool has = lane_pair<N>(g, step, p, q);
    int sw;
    if constexpr (LN <= 32) {
        sw = jacobi_v32<N>(A32, V32, g, group_mask<LN>(), pair_mask, keep);
        grp.sync();
    } else {
        sw = jacobi_v32_team<N, false>(A32, V32, reinterpret_cast<C<float>*>(V), reinterpret_cast<float*>(nrm), g, grp, pair_mask,
                                keep);
        grp.sync();
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) V[g + j * LN] = ccast<double>(V32[g + j * LN]);
    grp.sync();
    half_defect32<N>(V32, A32, g, grp, has, p, q);
    add_product32<N>(V, V32, A32, g, grp);
    if constexpr (F64) {
        const C<double> e = gram<N>(V, nrm, g, grp, has, p, q);
        if (has) {
            const C<float> ef = ccast<float>(-0.5 * e);
            A32[q * N + p] = ef;
            A32[p * N + q] = conj(ef);
        }
        if (g < N) A32[g * N + g] = C<float>{(float)fma(-0.5, nrm[g], 0.5), 0.f};
        grp.sync();
        add_product32<N>(V, V32, A32, g, grp);
    }
    return sw;
}

// On exit A holds U S (columns unsorted), V the right singular vectors and nrm the squared
// column norms of A.  keep_rank, cut: the caller keeps at most keep_rank singular triplets and
// drops those at or below cut times the largest; only pairs with a column among the keep_rank
// largest (norms within a factor 4 of the keep_rank-th count) and above cut / 2 are brought to
// orthogonality, judged against the larger column when the other one is not kept.  A32, V32
// (N^2 complex floats), T (N^2 complex) and relmask (one word) are scratch; the group has
// N^2 / 2 lanes.
template <int N, bool F64, typename Group>
__device__ SvdCount refined_svd(C<double>* A, C<double>* V, C<float>* A32, C<float>* V32, C<double>* T, double* nrm,
                                unsigned* relmask, int g, const Group& grp, unsigned pair_mask, double cut,
                                int keep_rank, float stop, double tol) {
    using CD = C<double>;
    using CF = C<float>;
    constexpr int LN = N * N / 2, NP = N * (N - 1) / 2, MAXP = 8;
    constexpr float KMAX2 = 1e-8f;   // |K|^2 limit of the simultaneous rotations
    SvdCount cnt;
    int step, p, q;
    const bool has = lane_pair<N>(g, step, p, q);
    {
        int e = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const CD a = A[g + j * LN];
            e = max(e, max(exp_bits(a.x), exp_bits(a.y)));
        }
        const double sc = inv_exp2(grp.max_int(e));
#pragma unroll
        for (int j = 0; j < 2; ++j) A32[g + j * LN] = ccast<float>(sc * A[g + j * LN]);
        grp.sync();
    }
    cnt.sweeps32 = svd32_unitary<N, F64>(V, A32, V32, nrm, g, grp, pair_mask, keep_rank);
    mul64<N, false>(A, V, g, grp);
    const float stop2 = stop * stop, cut2 = (float)(0.25 * cut * cut), tol2 = (float)(tol * tol);
    constexpr float OPEN2 = F64 ? 1e-16f : KMAX2;
    int second = 0;   // FP32 runs on a part of the columns
    for (int pass = 0;; ++pass) {
        const CD gam = gram<N>(A, nrm, g, grp, has, p, q);
        ++cnt.passes;
        cnt.pairs += NP;
        CF K = CF{0.f, 0.f};
        // 1: an open pair, 2: one of those with a large K, 32: and with a cosine above stop, 4: |K| > 1e-8,
        // 8: any K, 16: a K that moves the pair's shorter column by more than 1e-3 of its length; from bit 8 on:
        // sizes of K and c (below)
        unsigned flags = 0u;
        // F64: which columns of the pair count, their difference (scaled by the longer one), that scale
        // against the longest column's, and the product of two columns that do not count
        bool rp = false, rq = false;
        float dn = 0.f;
        int down = 0;
        CF cross = CF{0.f, 0.f};
        if (has) {
            const double al = nrm[p], be = nrm[q];
            // the upper words of positive doubles compare as integers; + 2 in the exponent: times 4
            const int ha = __double2hiint(al), hb = __double2hiint(be), a4 = ha + (2 << 20), b4 = hb + (2 << 20);
            int hmax = 0, next = INT_MAX;   // longest column; shortest one clearly longer than the pair's
            int ca = 0, cb = 0;
            for (int j = 0; j < N; ++j) {
                const int x = __double2hiint(nrm[j]);
                ca += x > a4;
                cb += x > b4;
                hmax = max(hmax, x);
                if (F64) next = x > max(a4, b4) ? min(next, x) : next;
            }
            const double sc = inv_exp2(max(ha, hb) >> 20);
            const float an = (float)(al * sc), bn = (float)(be * sc);
            const float top = (float)(__hiloint2double(hmax, 0) * sc);
            rp = ca < keep_rank && an >= cut2 * top;
            rq = cb < keep_rank && bn >= cut2 * top;
            down = (hmax >> 20) - (max(ha, hb) >> 20);
            const double gsc = sc * 1073741824.0;   // gamma times 2^30: |gamma|^2 stays in the FP32 range
            const float gx = (float)(gam.x * gsc), gy = (float)(gam.y * gsc);
            const float g2 = fmaf(gx, gx, gy * gy);
            if ((rp || rq) && sc > 0.0) {
                dn = (float)((be - al) * sc);
                const float lim = rp && rq ? an * bn : fmaxf(an, bn) * fmaxf(an, bn);
                const bool wide = g2 > stop2 * 1.152921504606847e18f * lim;
                if (wide) flags |= 1u;
                if (g2 > 0.f) {
                    const float g2n = g2 * 8.673617379884035e-19f;
                    const float tn = 2.f * 9.313225746154785e-10f * __frcp_rn(fabsf(dn) + sqrtf(fmaf(dn, dn, 4.f * g2n)));
                    const float t = dn >= 0.f ? tn : -tn;
                    K = CF{t * gx, t * gy};
                    const float k2 = norm2(K);
                    // Columns of nearly the same length: the rotation is gamma over the difference of the
                    // squared lengths, which may be of order one where the cosine is far below `stop`
                    // (a cosine of 1e-9 between lengths equal to 1e-9 leaves the kept triplets open).  Such a
                    // pair is open until K is small or the cosine is rounding.
                    const bool above = g2 > tol2 * 1.152921504606847e18f * lim;
                    if (k2 > OPEN2 && above) flags |= 1u;
                    // bit 8 + i: a |K| of at least 2^(-30 - 3 i) between a column that counts and another one
                    if (F64 && above && !(rp && rq)) {
                        const int i = max(0, (72 - (__float_as_int(k2) >> 23)) / 6);
                        if (i < 8) flags |= (0xffu << i & 0xffu) << 8;
                    }
                    if (!(k2 <= KMAX2)) {
                        K = CF{0.f, 0.f};
                        if (flags & 1u) flags |= wide ? 34u : 2u;
                    } else {
                        flags |= 8u;
                        if (k2 > 1e-16f) flags |= 4u;
                        if (k2 * fmaxf(an, bn) > 1e-6f * fminf(an, bn) && (rp && rq)) flags |= 16u;
                    }
                }
            } else if (F64) {
                // two columns that do not count, and c, their product over the squared length of the shortest
                // column that is clearly longer (exponents only): bit 16 + i for c of at least 2^(-20 + 3 i),
                // bit 24 + i for c^2
                const int e = (__float_as_int(g2) >> 23) - 187 - 2 * ((next >> 20) - (max(ha, hb) >> 20));
                if (e >= -40) flags |= ((1u << min((e + 46) / 6, 8)) - 1u) << 16;
                if (e >= -20) flags |= ((1u << min((e + 23) / 3, 8)) - 1u) << 24;
                const float f = __int_as_float(max(127 - down, 0) << 23);
                cross = CF{f * gx, f * gy};
            }
        }
        unsigned mine = flags;
        flags = grp.or_bits(flags);
        // A rotation K of a column that counts against one of those two leaves K c against the other, so a
        // pass would gain a factor c there instead of squaring.  Where K c is above rounding (about 2^-50)
        // the rotations take that term along (below), which leaves K c^2; open while that is above
        // rounding, and from the fourth pass on two such columns with c above 2^-11 are rotated themselves.
        // (Further passes alone instead: 2.19 passes per gate for 2.11, FP64 anneals 2 to 4 % longer.)
        const bool coupled = F64 && ((flags >> 8) & (flags >> 16) & 0xffu);
        if (F64 && ((flags >> 8) & (flags >> 24) & 0xffu)) {
            const bool late = pass >= 3;
            flags |= late && (flags & 1u << 19) ? 3u : 1u;
            if (late && (mine & 1u << 19)) mine |= 2u;
        }
        if (flags & 8u) {
            // I + K + K^2/2 on W (FP64) and V (FP64, or the correction in FP32)
            if (has) {
                A32[q * N + p] = K;
                A32[p * N + q] = CF{-K.x, K.y};
            }
            if (g < N) A32[g * N + g] = CF{0.f, 0.f};
            if (coupled) {
                // K_qp of a kept column p and another one q solves gamma_qp + (|a_q|^2 - |a_p|^2) K_qp +
                // sum_r a_q^H a_r K_rp = 0, r over the others: one step of that sum from the K above.  Only
                // where q is clearly the shorter one, as it is against every column that is kept (two equal
                // columns may lie on both sides of the line between those that count and the others)
                if (has) {
                    V32[q * N + p] = cross;
                    V32[p * N + q] = conj(cross);
                }
                if (g < N) V32[g * N + g] = CF{0.f, 0.f};
                grp.sync();
                if (rp != rq && fabsf(dn) > 0.5f && norm2(K) > 0.f) {
                    const int kept = rp ? p : q, other = rp ? q : p;
                    CF sum = CF{0.f, 0.f};
                    for (int r = 0; r < N; ++r) sum = cfma(V32[r * N + other], A32[kept * N + r], sum);
                    const float f = __int_as_float(min(97 + down, 254) << 23) / (rp ? -dn : dn);
                    const CF next = rp ? K - conj(f * sum) : K + f * sum;
                    if (norm2(next) <= KMAX2) K = next;
                }
                grp.sync();
                if (has) {
                    A32[q * N + p] = K;
                    A32[p * N + q] = CF{-K.x, K.y};
                }
            }
            grp.sync();
            CF l[2];
            // mixed mode: the corrections W L and V L in FP32, whose rounding is then below 1e-10 of every
            // kept column (its storage is complex64); else in FP64
            const bool low = !F64 && !(flags & 16u);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int t = g + j * LN, c = t / N, r = t % N;
                const CF k1 = A32[t];
                CF k2 = CF{0.f, 0.f};
                if (flags & 4u)
                    for (int s = 0; s < N; ++s) k2 = cfma(A32[s * N + r], A32[c * N + s], k2);
                l[j] = k1 + 0.5f * k2;
                if (!low) {
                    CD x = ccast<double>(k1);
                    if (flags & 4u) x = x + ccast<double>(0.5f * k2);
                    T[t] = x;
                }
            }
            grp.sync();
            if (!low) mul64<N, true>(A, T, g, grp);
            if (F64 && (flags & 4u)) {
                mul64<N, true>(V, T, g, grp);
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    A32[g + j * LN] = l[j];
                    if constexpr (F64) V32[g + j * LN] = ccast<float>(V[g + j * LN]);
                }
                grp.sync();
                if (low) correct32<N>(A, reinterpret_cast<CF*>(T), A32, g, grp);
                add_product32<N>(V, V32, A32, g, grp);
            }
        }
        if (!(flags & 1u)) break;
        if (pass + 1 >= MAXP) {
            int nsteps = 0;
            // to the resolution of the rotations: `stop` would leave pairs of close lengths open
            cnt.passes += jacobi_polish<N>(A, V, nrm, g, grp, pair_mask, tol, 16.0 * tol, 60, &cnt.rot, keep_rank,
                                                        relmask, &nsteps);
            cnt.pairs += nsteps * (N / 2);
            break;
        }
        if (!(flags & 2u)) continue;
        const unsigned steps = grp.or_bits((mine & 2u) ? 1u << step : 0u);
        const int nst = __popc(steps);
        bool part = false;
        if constexpr (N >= 16)   // FP32 resolves nothing below a cosine of 1e-7
            part = second < 3 && __popc(grp.or_bits((mine & 32u) ? 1u << step : 0u)) > N / 4;
        if (!part) {
            jacobi_polish<N>(A, V, nrm, g, grp, pair_mask, tol, stop, 1, &cnt.rot, N, nullptr, nullptr, steps);
            cnt.pairs += nst * (N / 2);
        } else if constexpr (N >= 16) {
            ++second;
            // the columns of those pairs, and every shorter one
            unsigned cols = grp.or_bits((mine & 32u) ? (1u << p) | (1u << q) : 0u);
            double longest = 0.0;
            for (int j = 0; j < N; ++j)
                if ((cols >> j) & 1u) longest = fmax(longest, nrm[j]);
            for (int j = 0; j < N; ++j) cols |= nrm[j] <= longest ? 1u << j : 0u;
            grp.sync();
            int e = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const CD a = A[g + j * LN];
                if ((cols >> ((g + j * LN) / N)) & 1u) e = max(e, max(exp_bits(a.x), exp_bits(a.y)));
            }
            const double sc = inv_exp2(grp.max_int(e));
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int t = g + j * LN;
                A32[t] = ((cols >> (t / N)) & 1u) ? ccast<float>(sc * A[t]) : CF{0.f, 0.f};
            }
            grp.sync();
            cnt.sweeps32 += svd32_unitary<N, F64>(T, A32, V32, nrm, g, grp, pair_mask, N);
            mul64<N, false>(A, T, g, grp);
            mul64<N, false>(V, T, g, grp);
        }
        if constexpr (!F64) {
#pragma unroll
            for (int j = 0; j < 2; ++j) V32[g + j * LN] = ccast<float>(V[g + j * LN]);
            grp.sync();
        }
    }
    column_norms<N>(A, nrm, g);
    grp.sync();
    return cnt;
}

// Rank of value i among n values, descending, ties by index (used to sort
// singular values without data movement).  A NaN ranks below every number, so the
// ranks are a permutation of 0..n-1 whatever the values.
template <typename R>
__device__ __forceinline__ int desc_rank(const R* v, int n, int i) {
    const R x0 = v[i];
    const R x = (x0 == x0) ? x0 : (R)-INFINITY;
    int rk = 0;
    for (int j = 0; j < n; ++j) {
        const R y0 = v[j];
        const R y = (y0 == y0) ? y0 : (R)-INFINITY;
        rk += (y > x) || (y == x && j < i);
    }
    return rk;
}

// desc_rank for non-negative doubles on the integer pipe (their bits order as integers; a NaN
// ranks below every number).
__device__ __forceinline__ int desc_rank_bits(const double* v, int n, int i) {
    constexpr long long inf = 0x7ff0000000000000ll;
    const long long x0 = __double_as_longlong(v[i]), x = x0 >= 0 && x0 <= inf ? x0 : -1;
    int rk = 0;
    for (int j = 0; j < n; ++j) {
        const long long y0 = __double_as_longlong(v[j]), y = y0 >= 0 && y0 <= inf ? y0 : -1;
        rk += (y > x) || (y == x && j < i);
    }
    return rk;
}

}  // namespace gtqa

namespace gtqa {

// ---------------------------------------------------------------------------
// Teams of TEAM threads inside a block: TEAM <= 32 lives in one warp (warp-level
// sync with the team's lane mask); TEAM a multiple of 32 syncs with named barrier
// 1 + team id (barrier 0 stays free for __syncthreads).
// ---------------------------------------------------------------------------
template <int TEAM>
__device__ __forceinline__ void team_bar(int team) {
    if constexpr (TEAM <= 32) {
        __syncwarp(group_mask<TEAM>());
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(TEAM) : "memory");
    }
}

// Synchronisation policy for a multi-warp team (named barrier + shared flag).
template <int TEAM>
struct TeamGroup {
    int team;
    int* flag;
    __device__ __forceinline__ void sync() const { team_bar<TEAM>(team); }
    __device__ __forceinline__ bool any(int p) const {
        team_bar<TEAM>(team);
        if ((threadIdx.x % TEAM) == 0) *flag = 0;
        team_bar<TEAM>(team);
        if (p) atomicOr(flag, 1);
        team_bar<TEAM>(team);
        return *(volatile int*)flag != 0;
    }
    __device__ __forceinline__ int max_int(int v) const {
        team_bar<TEAM>(team);
        if ((threadIdx.x % TEAM) == 0) *flag = INT_MIN;
        team_bar<TEAM>(team);
        atomicMax(flag, v);
        team_bar<TEAM>(team);
        return *(volatile int*)flag;
    }
    __device__ __forceinline__ unsigned or_bits(unsigned v) const {
        team_bar<TEAM>(team);
        if ((threadIdx.x % TEAM) == 0) *flag = 0;
        team_bar<TEAM>(team);
        if (v) atomicOr(reinterpret_cast<unsigned*>(flag), v);
        team_bar<TEAM>(team);
        return *reinterpret_cast<volatile unsigned*>(flag);
    }
};

// L2-coherent loads for data written by other blocks during the same launch.
template <typename T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }
template <>
__device__ __forceinline__ C<double> ldcg(const C<double>* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return C<double>{v.x, v.y};
}
template <>
__device__ __forceinline__ C<float> ldcg(const C<float>* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return C<float>{v.x, v.y};
}

// ---------------------------------------------------------------------------
// Grid-wide barrier for a cooperative (co-resident) launch.  Sense reversal on a
// generation counter; the wait is bounded: after `limit` polls the block records
// GTQA timeout in *err and leaves.  Callers test *err after every barrier and
// return, so a lost block can never hang the device.
// ---------------------------------------------------------------------------
// Grid barrier for cooperative launches over a monotonic 64-bit arrival counter: the
// k-th barrier of a launch completes when the counter reaches base + k * nblocks, so
// an arrival is one release-atomic and the wait one acquire-load poll, with no
// separate generation word to publish.  Thread 0 of each block keeps the target.  Every
// wait is bounded: after `limit` polls the block records GTQA_ERR_TIMEOUT in *err and
// leaves (the others then time out at this or their next barrier).  Launches must pass
// the same number of barriers in every block, which keeps the counter at a multiple of
// nblocks between launches.
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long atom_add_release_u64(unsigned long long* p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.add.release.gpu.global.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

struct GridBarrier {
    unsigned long long* count;
    int* err;
    unsigned long long next;   // thread 0: counter value that completes the next barrier
    unsigned int nblocks;
};

__device__ __forceinline__ GridBarrier grid_barrier_init(unsigned long long* count, int* err, unsigned int nblocks) {
    GridBarrier gb{count, err, 0ull, nblocks};
    if (threadIdx.x == 0) {
        // at most nblocks - 1 blocks can have arrived at this launch's first barrier
        const unsigned long long c = *(volatile unsigned long long*)count;
        gb.next = c - c % nblocks + nblocks;
    }
    return gb;
}

__device__ __forceinline__ bool grid_sync(GridBarrier& gb, long long limit) {
    __shared__ int ok_shared;
    __syncthreads();   // the block's writes happen before thread 0's release
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned long long old = atom_add_release_u64(gb.count, 1ull);
        if (old + 1ull < gb.next) {
            long long polls = 0;
            while (ld_acquire_u64(gb.count) < gb.next) {
                if (++polls > limit) {
                    atomicExch(gb.err, 6);   // GTQA_ERR_TIMEOUT
                    ok = 0;
                    break;
                }
                if (polls > 2048) __nanosleep(32);
            }
        }
        gb.next += gb.nblocks;
        ok_shared = ok;
    }
    __syncthreads();
    return ok_shared != 0;   // one value per block, so the whole block leaves together
}

// grid_sync with a step of the first warp between the block's barrier and its arrival: pre()
// runs on warp 0 once the block's shared-memory writes are visible to it, and thread 0's
// release arrival follows in program order, so what pre() writes to global memory is visible
// to every block that passes this barrier.
template <class Pre>
__device__ __forceinline__ bool grid_sync_pre(GridBarrier& gb, long long limit, Pre&& pre) {
    __shared__ int ok_pre;
    __syncthreads();
    if (threadIdx.x < 32) {
        pre();
        __syncwarp();
    }
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned long long old = atom_add_release_u64(gb.count, 1ull);
        if (old + 1ull < gb.next) {
            long long polls = 0;
            while (ld_acquire_u64(gb.count) < gb.next) {
                if (++polls > limit) {
                    atomicExch(gb.err, 6);   // GTQA_ERR_TIMEOUT
                    ok = 0;
                    break;
                }
                if (polls > 2048) __nanosleep(32);
            }
        }
        gb.next += gb.nblocks;
        ok_pre = ok;
    }
    __syncthreads();
    return ok_pre != 0;
}

// The dynamic shared-memory limit is an attribute of the kernel function, shared by
// every state in the process, while the BP kernel's need grows with the number of
// instances.  The limit is therefore raised to the device maximum (not to one state's
// need), so that states of different sizes can launch the same kernel in any order.
template <class K>
inline cudaError_t raise_smem_limit(K kernel, size_t smem) {
    int dev = 0, mx = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    const size_t avail = (size_t)mx > fa.sharedSizeBytes ? (size_t)mx - fa.sharedSizeBytes : 0;
    if (smem > avail) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)avail);
}

}  // namespace gtqa
