// The plain path: graph tensor networks whose vertex tensors are too large or have too many
// bonds for the persistent kernels, or that run every step in FP32.  Shapes built: degree 4
// with CHI <= 4 (the random 4-regular graphs of Sec. V) and degree 3 with CHI = 16 (the largest
// bond dimension of the chi sweep), in complex128 (the FP64 precision mode, R = RC = double) and
// in the mixed mode (complex64 storage and contractions, R = float, with the normalisation,
// trace norms, regauge and the CHI = 16 gate's QR/SVD in RC = double); degree 3 with CHI <= 8 or
// CHI = 16 and degree 4 with CHI <= 4 in complex64 with every step in FP32 (the complex64 mode,
// R = RC = float).  One instance.  The messages hold m itself in FP64 and complex64 and, as on
// the persistent path, delta = m - m0 with m0 = diag(lambda)/sum(lambda) in the mixed mode
// (BP contracts only the delta terms in FP32; the warm-start defect D0 is computed in FP64 and
// stored in complex64, its trace t0 in complex128).
//
// Layout: Gamma and T are [n][2][CHI]^D (slot k = k-th incident edge in ascending id, stride
// CHI^(D-1-k); phantom slots of vertices with fewer edges have dimension 1 with lambda = e_0);
// lambda [m][CHI]; messages [2m][CHI][CHI] as in the persistent path.
// The steps are those of the persistent path, in plain launches:
//   gates    one launch per colour: plain_ising_kernel (CHI <= 8), ising16_gate_kernel
//            (CHI = 16), the per-physical-index QR-reduced simple update with a 2 CHI x 2 CHI
//            core (App. E, App. D "Truncation"), the mixing gates (Sec. II D) fused;
//   bp       T = Gamma prod lambda^{1/2} (Eq. (symmetric_gauge)), warm start
//            diag(lambda)/sum(lambda) (Eq. (reconstructed_messages)); per flooding sweep of
//            Eq. (local_consistency) one launch over vertices and one over messages for the
//            exact trace-norm distance (App. B); the host reads the distance after every sweep;
//   regauge  per edge the Vidal gauge transforms from the two messages (App. D "Vidal gauge
//            finding"), then per vertex the transforms applied to T;
//   marginals  Eq. (partial_dens) with the environment of Eq. (bp_approx);
//   residual   R of App. C per (vertex, slot), FP64 trace norms (the regauge policy of
//              Sec. II C reads it on the host);
//   sampling   the projection step of Sec. IV A for one vertex, then BP and the regauge.
#pragma once

#include <type_traits>

#include "gtqa_general.cuh"

namespace gtqa {

struct PlainArgs {
    void* Gamma;
    void* T;
    double* lam;
    const void* msg_cur;      // incoming and previous outgoing messages
    void* msg_nxt;            // new outgoing messages
    void* X;                  // regauge transforms [m][2][CHI^2]
    void* dm;                 // [2m][CHI^2]: new - old of every outgoing message of a sweep
    void* scratch;            // per-block tensor buffers when shared memory is too small
    const int4* vslots;       // slots per vertex (x, y, z, w; -1 phantom)
    const int4* edge_info;    // (u, v, slot at u, slot at v)
    int n, m;
    double* acc;              // distance accumulator (one double)
    int warm;
    void* D0;                 // mixed mode: [2m][CHI^2] warm-start defect F(m0) - tr F(m0) m0 (storage type)
    cd* t0;                   // mixed mode: [2m] tr F(m0)
};

template <int CHI, int D, typename R = double>
struct PlainShape {
    static constexpr int H = ipow(CHI, D), H2 = 2 * H, CC = CHI * CHI;
    static constexpr int NT = 16 * CC < 1024 ? 16 * CC : 1024;    // threads of the sweep kernel
    static constexpr int TPO = NT / CC;                           // threads per message entry
    static constexpr bool SMEM = 3 * H2 * (int)sizeof(C<R>) <= 48 * 1024;   // tensor buffers in shared memory
    static constexpr size_t scratch_per_block = SMEM ? 0 : (size_t)3 * H2;   // complex entries
};

__device__ __forceinline__ int plain_slot_edge(const int4& v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}

// T = Gamma prod_k lambda_k^{1/2}; with warm, the vertex's outgoing messages are set to
// diag(lambda)/sum(lambda) in msg_nxt (the buffer the first sweep reads).  One block per vertex.
template <int CHI, int D, typename R, typename RC = R>
__global__ void plain_bp_init_kernel(PlainArgs a) {
    using S = PlainShape<CHI, D, R>;
    const int v = blockIdx.x;
    __shared__ RC sq[D][CHI], m0[D][CHI];
    const int4 sl = a.vslots[v];
    if (threadIdx.x < D * CHI) {
        const int k = threadIdx.x / CHI, j = threadIdx.x % CHI;
        const int e = plain_slot_edge(sl, k);
        const RC lj = lam_get(a.lam, CHI, e, j);
        sq[k][j] = sqrt(lj);
        RC s = 0.0;
        for (int q = 0; q < CHI; ++q) s += lam_get(a.lam, CHI, e, q);
        m0[k][j] = s > 0.0 ? lj / s : 0.0;
    }
    __syncthreads();
    const C<R>* g = (const C<R>*)a.Gamma + (size_t)v * S::H2;
    C<R>* T = (C<R>*)a.T + (size_t)v * S::H2;
    for (int t = threadIdx.x; t < S::H2; t += blockDim.x) {
        int r = t % S::H;
        RC f = 1.0;
        for (int k = D - 1; k >= 0; --k) {
            f *= sq[k][r % CHI];
            r /= CHI;
        }
        T[t] = ccast<R>(f * ccast<RC>(g[t]));
    }
    constexpr bool MIX = sizeof(R) != sizeof(RC);
    if (a.warm) {
        // the mixed mode holds delta = m - m0, which the warm start sets to 0
        C<R>* out = (C<R>*)a.msg_nxt;
        for (int t = threadIdx.x; t < D * S::CC; t += blockDim.x) {
            const int k = t / S::CC, r = t % S::CC;
            const int e = plain_slot_edge(sl, k);
            if (e < 0) continue;
            const int o = 2 * e + (a.edge_info[e].x == v ? 0 : 1);
            const int j = r / CHI, jp = r % CHI;
            out[(size_t)o * S::CC + r] = C<R>{(!MIX && j == jp) ? (R)m0[k][j] : (R)0, (R)0};
        }
    }
    if constexpr (MIX) {
        // F0 = F(m0) of every outgoing message in RC from the stored T (so that F(m0 + delta) =
        // F0 + F_delta holds for the T the sweeps contract), kept as D0 = F0 - tr(F0) m0 and t0
        __shared__ C<RC> F0[D][S::CC];
        __shared__ C<RC> tr0[D];
        __syncthreads();   // this block's T is written
        constexpr int NO = S::H / CHI;
        for (int t = threadIdx.x; t < D * S::CC; t += blockDim.x) {
            const int k = t / S::CC, r = t % S::CC;
            if (plain_slot_edge(sl, k) < 0) continue;
            const int j = r / CHI, jp = r % CHI;
            int sk = 1;
            for (int l = D - 1; l > k; --l) sk *= CHI;
            C<RC> f = C<RC>{(RC)0, (RC)0};
            for (int i = 0; i < 2; ++i)
                for (int q = 0; q < NO; ++q) {
                    int rem = q, base = 0, stride = 1;
                    RC w = 1.0;
                    for (int l = D - 1; l >= 0; --l) {
                        if (l != k) {
                            const int idx = rem % CHI;
                            rem /= CHI;
                            w *= m0[l][idx];
                            base += idx * stride;
                        }
                        stride *= CHI;
                    }
                    const C<RC> x = ccast<RC>(T[i * S::H + base + j * sk]), y = ccast<RC>(T[i * S::H + base + jp * sk]);
                    f = cfmac(y, w * x, f);
                }
            F0[k][r] = f;
        }
        __syncthreads();
        if (threadIdx.x < D) {
            C<RC> tr = C<RC>{(RC)0, (RC)0};
            for (int j = 0; j < CHI; ++j) tr = tr + F0[threadIdx.x][j * CHI + j];
            tr0[threadIdx.x] = tr;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < D * S::CC; t += blockDim.x) {
            const int k = t / S::CC, r = t % S::CC;
            const int e = plain_slot_edge(sl, k);
            if (e < 0) continue;
            const int o = 2 * e + (a.edge_info[e].x == v ? 0 : 1);
            const int j = r / CHI, jp = r % CHI;
            C<RC> d = F0[k][r];
            if (j == jp) d = d - m0[k][j] * tr0[k];
            ((C<R>*)a.D0)[(size_t)o * S::CC + r] = ccast<R>(d);
            if (r == 0) a.t0[o] = ccast<double>(tr0[k]);
        }
    }
}

// One flooding sweep for one vertex: every outgoing message
//   m_{v->b}[j][j'] = sum T[.., j@s, ..] conj(T[.., j'@s, ..]) prod_{o != s} m_o[x_o][x'_o]
// (Eq. (local_consistency)), divided by its complex trace; new - old goes to dm for the
// trace-norm kernel.
// R is the storage and contraction type; RC the type of the trace and the normalisation
// (FP64 in the mixed mode).
template <int CHI, int D, typename R, typename RC = R>
__global__ void __launch_bounds__(PlainShape<CHI, D, R>::NT) plain_bp_sweep_kernel(PlainArgs a) {
    using S = PlainShape<CHI, D, R>;
    constexpr int H2 = S::H2, CC = S::CC, NT = S::NT, TPO = S::TPO;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    C<R>* min = reinterpret_cast<C<R>*>(plain_smem);   // [D][CC]
    C<R>* F = min + D * CC;                          // [CC]
    C<R>* T;
    C<R>* P0;
    C<R>* P1;
    if constexpr (S::SMEM) {
        T = F + CC;
        P0 = T + H2;
        P1 = P0 + H2;
    } else {
        T = (C<R>*)a.scratch + (size_t)blockIdx.x * S::scratch_per_block;
        P0 = T + H2;
        P1 = P0 + H2;
    }
    __shared__ int es[4], in_idx[4], out_idx[4];
    __shared__ C<RC> itr;
    // mixed mode (the delta form of the persistent path): the messages hold delta = m - m0 with
    // m0 = diag(lambda)/sum(lambda); mz and md hold m0 and delta of the incoming messages
    constexpr bool MIX = sizeof(R) != sizeof(RC);
    C<R>* mz = min + (D + 1) * CC + (S::SMEM ? 3 * H2 : 0);   // [D][CC], mixed mode only
    C<R>* md = mz + D * CC;                                  // [D][CC], mixed mode only
    __shared__ RC m0d[D][CHI];
    __shared__ C<RC> tau;
    const int v = blockIdx.x, tid = threadIdx.x;
    const C<R>* src_msg = (const C<R>*)a.msg_cur;
    C<R>* dst_msg = (C<R>*)a.msg_nxt;
    if (tid < D) {
        const int e = plain_slot_edge(a.vslots[v], tid);
        es[tid] = e;
        if (e >= 0) {
            const bool first = a.edge_info[e].x == v;
            out_idx[tid] = 2 * e + (first ? 0 : 1);
            in_idx[tid] = 2 * e + (first ? 1 : 0);
        } else {
            out_idx[tid] = in_idx[tid] = -1;
        }
    }
    if (MIX && tid < D * CHI) {
        const int k = tid / CHI, j = tid % CHI;
        const int e = plain_slot_edge(a.vslots[v], k);
        RC sum = 0.0;
        for (int q = 0; q < CHI; ++q) sum += lam_get(a.lam, CHI, e, q);
        m0d[k][j] = sum > 0.0 ? lam_get(a.lam, CHI, e, j) / sum : 0.0;
    }
    for (int t = tid; t < H2; t += NT) T[t] = ((const C<R>*)a.T)[(size_t)v * H2 + t];
    __syncthreads();
    for (int t = tid; t < D * CC; t += NT) {
        const int k = t / CC, r = t % CC;
        if constexpr (MIX) {
            const int j = r / CHI, jp = r % CHI;
            const C<R> dv = in_idx[k] >= 0 ? src_msg[(size_t)in_idx[k] * CC + r] : C<R>{(R)0, (R)0};
            const C<R> zv = C<R>{j == jp ? (R)m0d[k][j] : (R)0, (R)0};
            md[t] = dv;
            mz[t] = zv;
            min[t] = zv + dv;
        } else {
            min[t] = in_idx[k] >= 0 ? src_msg[(size_t)in_idx[k] * CC + r] : C<R>{(R)(r == 0 ? 1 : 0), (R)0};
        }
    }
    __syncthreads();
    if constexpr (MIX) {
        // F(m0 + delta) - F(m0) telescoped over the other slots o_1 < o_2 < ...: chain c takes
        // m0 on the slots before its own, delta on its own and m after it (FP32 contractions);
        // then delta' = (D0 + F_delta - m0 tr F_delta) / (t0 + tr F_delta) in RC
        for (int s = 0; s < D; ++s) {
            if (es[s] < 0) continue;   // uniform: es is shared
            const int ss = ipow(CHI, D - 1 - s);
            constexpr int NTERM = H2 / CHI;
            for (int c = 0; c < D - 1; ++c) {
                const C<R>* src = T;
                C<R>* dst = P0;
                int i = 0;
                for (int o = 0; o < D; ++o) {
                    if (o == s) continue;
                    const C<R>* mo = (i < c ? mz : (i == c ? md : min)) + o * CC;
                    ++i;
                    const int so = ipow(CHI, D - 1 - o);
                    for (int t = tid; t < H2; t += NT) {
                        const int x = (t / so) % CHI, base = t - x * so;
                        C<R> acc = C<R>{(R)0, (R)0};
#pragma unroll 4
                        for (int q = 0; q < CHI; ++q) acc = cfma(src[base + q * so], mo[q * CHI + x], acc);
                        dst[t] = acc;
                    }
                    __syncthreads();
                    src = dst;
                    dst = (dst == P0) ? P1 : P0;
                }
                for (int rr = tid / TPO; rr < CC; rr += NT / TPO) {
                    const int part = tid % TPO;
                    const int j = rr / CHI, jp = rr % CHI;
                    C<R> f = C<R>{(R)0, (R)0};
                    for (int q = part; q < NTERM; q += TPO) {
                        const int t = (q / ss) * (ss * CHI) + (q % ss);
                        f = cfmac(T[t + jp * ss], src[t + j * ss], f);
                    }
                    f.x = group_sum<TPO>(f.x, group_mask<TPO>());
                    f.y = group_sum<TPO>(f.y, group_mask<TPO>());
                    if (part == 0) F[rr] = c == 0 ? f : F[rr] + f;
                }
                __syncthreads();
            }
            const int out = out_idx[s];
            if (tid == 0) {
                C<RC> tr = C<RC>{(RC)0, (RC)0};
                for (int q = 0; q < CHI; ++q) tr = tr + ccast<RC>(F[q * CHI + q]);
                tau = tr;
                const C<RC> den = a.t0[out] + tr;
                const RC d = den.x * den.x + den.y * den.y;
                itr = d > 0.0 ? C<RC>{den.x / d, -den.y / d} : C<RC>{(RC)0, (RC)0};
            }
            __syncthreads();
            for (int r = tid; r < CC; r += NT) {
                const int j = r / CHI, jp = r % CHI;
                C<RC> num = ccast<RC>(((const C<R>*)a.D0)[(size_t)out * CC + r]) + ccast<RC>(F[r]);
                if (j == jp) num = num - m0d[s][j] * tau;
                const C<RC> dn = num * itr;
                const C<RC> dold = ccast<RC>(src_msg[(size_t)out * CC + r]);
                dst_msg[(size_t)out * CC + r] = ccast<R>(dn);
                ((C<R>*)a.dm)[(size_t)out * CC + r] = ccast<R>(dn - dold);
            }
            __syncthreads();
        }
        return;
    }
    for (int s = 0; s < D; ++s) {
        if (es[s] < 0) continue;   // uniform: es is shared
        const C<R>* src = T;
        C<R>* dst = P0;
        for (int o = 0; o < D; ++o) {
            if (o == s) continue;
            const int so = ipow(CHI, D - 1 - o);
            for (int t = tid; t < H2; t += NT) {
                const int x = (t / so) % CHI, base = t - x * so;
                C<R> acc = C<R>{(R)0, (R)0};
#pragma unroll 4
                for (int q = 0; q < CHI; ++q) acc = cfma(src[base + q * so], min[o * CC + q * CHI + x], acc);
                dst[t] = acc;
            }
            __syncthreads();
            src = dst;
            dst = (dst == P0) ? P1 : P0;
        }
        // F[j][j'] = sum over the entries with slot-s index j of conj(T[.. j' ..]) src[.. j ..]
        const int ss = ipow(CHI, D - 1 - s);
        constexpr int NTERM = H2 / CHI;
        for (int rr = tid / TPO; rr < CC; rr += NT / TPO) {
            const int part = tid % TPO;
            const int j = rr / CHI, jp = rr % CHI;
            C<R> f = C<R>{(R)0, (R)0};
            for (int q = part; q < NTERM; q += TPO) {
                const int t = (q / ss) * (ss * CHI) + (q % ss);
                f = cfmac(T[t + jp * ss], src[t + j * ss], f);
            }
            f.x = group_sum<TPO>(f.x, group_mask<TPO>());
            f.y = group_sum<TPO>(f.y, group_mask<TPO>());
            if (part == 0) F[rr] = f;
        }
        __syncthreads();
        if (tid == 0) {
            C<RC> tr = C<RC>{(RC)0, (RC)0};
            for (int q = 0; q < CHI; ++q) tr = tr + ccast<RC>(F[q * CHI + q]);
            const RC d = tr.x * tr.x + tr.y * tr.y;
            itr = d > 0.0 ? C<RC>{tr.x / d, -tr.y / d} : C<RC>{(RC)0, (RC)0};
        }
        __syncthreads();
        for (int r = tid; r < CC; r += NT) {
            const C<RC> mn = ccast<RC>(F[r]) * itr;
            const C<RC> mo = ccast<RC>(src_msg[(size_t)out_idx[s] * CC + r]);
            dst_msg[(size_t)out_idx[s] * CC + r] = ccast<R>(mn);
            ((C<R>*)a.dm)[(size_t)out_idx[s] * CC + r] = ccast<R>(mn - mo);
        }
        __syncthreads();
    }
}

// Trace norm (sum of singular values, one-sided Jacobi in FP64) of every directed message's
// new - old; block = CHI^2 / 2 threads, one message per block; the sum goes to *acc.
template <int CHI, typename R, typename RC = R>
__global__ void plain_trace_norm_kernel(const C<R>* dm, double* acc) {
    constexpr int CC = CHI * CHI;
    __shared__ C<RC> A[CC];
    __shared__ RC tn;
    __shared__ int flag;
    const int g = threadIdx.x;
    for (int t = g; t < CC; t += blockDim.x) A[t] = ccast<RC>(dm[(size_t)blockIdx.x * CC + t]);
    if (g == 0) tn = 0.0;
    __syncthreads();
    BlockGroup grp{&flag};
    jacobi_svd<CHI, RC, BlockGroup, false>(A, nullptr, g, grp, group_mask<CHI>(), (RC)(sizeof(RC) == 8 ? 1e-15 : 1e-6),
                                           60, false);
    __syncthreads();
    if (g < CHI) {
        RC c2 = 0.0;
        for (int r = 0; r < CHI; ++r) c2 += norm2(A[g * CHI + r]);
        atomicAdd(&tn, sqrt(c2));
    }
    __syncthreads();
    if (g == 0) atomicAdd(acc, tn);
}

// Vidal gauge finding, edge part (App. D "Vidal gauge finding"), FP64, block = CHI^2 / 2
// threads: Hermitian eigen-decompositions of m_{a->b} and m_{b->a} (as SVDs; signs from
// v^H A v), principal square roots and pseudo-inverse square roots, the SVD of
// M = (m_{a->b}^{1/2})^T m_{b->a}^{1/2}, lambda = S/||S||, X_a = conj(m_{a->b}^{-1/2}) U ||S||^{1/2}
// and X_b = conj(m_{b->a}^{-1/2}) V^* ||S||^{1/2}.
template <int CHI, typename R, typename RC = R>
__global__ void plain_regauge_edge_kernel(const C<R>* msg, double* lam, C<R>* X, double eig_cut, double svd_cut) {
    constexpr int CC = CHI * CHI;
    __shared__ C<RC> Am[2][CC], Vm[2][CC], sqm[2][CC], isq[2][CC], M[CC], VM[CC];
    __shared__ RC w[2][CHI], sig[CHI], scal[2];
    __shared__ int perm[CHI], flag;
    const int e = blockIdx.x, tid = threadIdx.x, NT = blockDim.x;
    BlockGroup grp{&flag};
    // mixed mode: the messages hold delta = m - m0, m0 = diag(lambda_e)/sum(lambda_e) (read before
    // this kernel overwrites lambda_e)
    constexpr bool MIX = sizeof(R) != sizeof(RC);
    __shared__ RC m0e[CHI];
    if (MIX && tid < CHI) {
        RC sum = 0.0;
        for (int q = 0; q < CHI; ++q) sum += lam[(size_t)e * CHI + q];
        m0e[tid] = sum > 0.0 ? lam[(size_t)e * CHI + tid] / sum : 0.0;
    }
    if (MIX) __syncthreads();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC;
        const int row = r % CHI, col = r / CHI;
        const C<R>* mm = msg + (size_t)(2 * e + x) * CC;
        C<RC> v = ccast<RC>(mm[row * CHI + col]), vt = ccast<RC>(mm[col * CHI + row]);
        if (MIX && row == col) {
            v.x += m0e[row];
            vt.x += m0e[row];
        }
        Am[x][col * CHI + row] = C<RC>{(RC)0.5 * (v.x + vt.x), (RC)0.5 * (v.y - vt.y)};
    }
    __syncthreads();
    for (int x = 0; x < 2; ++x)
        jacobi_svd<CHI, RC, BlockGroup, true, sizeof(RC) == 8>(Am[x], Vm[x], tid, grp, group_mask<CHI>(),
                                                                  (RC)(sizeof(RC) == 8 ? 1e-15 : 1e-6), 60, true, nullptr,
                                                                  (RC)(sizeof(RC) == 8 ? 3e-8 : 1e-3));
    __syncthreads();
    for (int t = tid; t < 2 * CHI; t += NT) {
        const int x = t / CHI, k = t % CHI;
        RC n2 = 0.0, sg = 0.0;
        for (int r = 0; r < CHI; ++r) {
            const C<RC> av = Am[x][k * CHI + r], vv = Vm[x][k * CHI + r];
            n2 += norm2(av);
            sg += vv.x * av.x + vv.y * av.y;
        }
        const RC wv = nr_sqrt(n2);
        w[x][k] = sg >= 0.0 ? wv : -wv;
    }
    __syncthreads();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC;
        const int j = r / CHI, jp = r % CHI;
        RC wmax = 0.0;
        for (int k = 0; k < CHI; ++k) wmax = fmax(wmax, w[x][k]);
        C<RC> s1 = C<RC>{(RC)0, (RC)0}, s2 = C<RC>{(RC)0, (RC)0};
        for (int k = 0; k < CHI; ++k) {
            const RC wk = w[x][k];
            if (!(wk > eig_cut * wmax)) continue;
            const RC is = nr_rsqrt(wk);
            const RC sq = wk * is;
            const C<RC> vv = Vm[x][k * CHI + j] * conj(Vm[x][k * CHI + jp]);
            s1 = cfma(C<RC>{sq, (RC)0}, vv, s1);
            s2 = cfma(C<RC>{is, (RC)0}, vv, s2);
        }
        sqm[x][r] = s1;
        isq[x][r] = s2;
    }
    __syncthreads();
    for (int t = tid; t < CC; t += NT) {
        const int k = t % CHI, l = t / CHI;
        C<RC> acc = C<RC>{(RC)0, (RC)0};
        for (int j = 0; j < CHI; ++j) acc = cfma(sqm[0][j * CHI + k], sqm[1][j * CHI + l], acc);
        M[l * CHI + k] = acc;
    }
    __syncthreads();
    jacobi_svd<CHI, RC, BlockGroup, true, sizeof(RC) == 8>(M, VM, tid, grp, group_mask<CHI>(),
                                                         (RC)(sizeof(RC) == 8 ? 1e-15 : 1e-6), 60, true, nullptr,
                                                         (RC)(sizeof(RC) == 8 ? 3e-8 : 1e-3));
    __syncthreads();
    for (int cc = tid; cc < CHI; cc += NT) {
        RC n2 = 0.0;
        for (int r = 0; r < CHI; ++r) n2 += norm2(M[cc * CHI + r]);
        sig[cc] = nr_sqrt(n2);
    }
    __syncthreads();
    for (int cc = tid; cc < CHI; cc += NT) perm[desc_rank(sig, CHI, cc)] = cc;
    __syncthreads();
    if (tid == 0) {
        RC tot = 0.0;
        for (int cc = 0; cc < CHI; ++cc) tot += sig[cc] * sig[cc];
        const RC nrm = nr_sqrt(tot);
        scal[0] = nrm;
        scal[1] = nr_sqrt(nrm);
        const RC inrm = nrm > 0.0 ? nr_rcp(nrm) : 0.0;
        const RC smax = sig[perm[0]];
        for (int r = 0; r < CHI; ++r) {
            const RC s = sig[perm[r]];
            lam[(size_t)e * CHI + r] = (nrm > 0.0 && s > svd_cut * smax) ? s * inrm : 0.0;
        }
    }
    __syncthreads();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC;
        const int jpp = r / CHI, j = r % CHI;
        const int pc = perm[j];
        const RC s = sig[pc];
        C<RC> acc = C<RC>{(RC)0, (RC)0};
        const bool kept = scal[0] > 0.0 && s > svd_cut * sig[perm[0]];
        if (kept) {
            for (int jp = 0; jp < CHI; ++jp) {
                const C<RC> u = (x == 0) ? nr_rcp(s) * M[pc * CHI + jp] : conj(VM[pc * CHI + jp]);
                acc = cfma(isq[x][jp * CHI + jpp], u, acc);
            }
            acc = scal[1] * acc;
        }
        X[((size_t)e * 2 + x) * CC + r] = ccast<R>(acc);
    }
}

// Vidal gauge finding, vertex part: Gamma[.., j@k, ..] = sum_q T[.., q@k, ..] X_k[q][j] for every
// slot (X of the edge, from this vertex's side; identity on phantom slots).
template <int CHI, int D, typename R>
__global__ void plain_regauge_vertex_kernel(PlainArgs a) {
    using S = PlainShape<CHI, D, R>;
    constexpr int H2 = S::H2, CC = S::CC;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    C<R>* Xs = reinterpret_cast<C<R>*>(plain_smem);   // [D][CC]
    C<R>* b0;
    C<R>* b1;
    if constexpr (S::SMEM) {
        b0 = Xs + D * CC;
        b1 = b0 + H2;
    } else {
        b0 = (C<R>*)a.scratch + (size_t)blockIdx.x * S::scratch_per_block;
        b1 = b0 + H2;
    }
    const int v = blockIdx.x;
    const int4 sl = a.vslots[v];
    for (int t = threadIdx.x; t < H2; t += blockDim.x) b0[t] = ((const C<R>*)a.T)[(size_t)v * H2 + t];
    for (int t = threadIdx.x; t < D * CC; t += blockDim.x) {
        const int k = t / CC, r = t % CC;
        const int e = plain_slot_edge(sl, k);
        if (e >= 0) {
            const int side = a.edge_info[e].x == v ? 0 : 1;
            Xs[t] = ((const C<R>*)a.X)[((size_t)e * 2 + side) * CC + r];
        } else {
            Xs[t] = C<R>{(R)((r / CHI == r % CHI) ? 1 : 0), (R)0};
        }
    }
    __syncthreads();
    C<R>* cur = b0;
    C<R>* nxt = b1;
    for (int k = 0; k < D; ++k) {
        const int st = ipow(CHI, D - 1 - k);
        for (int t = threadIdx.x; t < H2; t += blockDim.x) {
            const int jk = (t / st) % CHI, base = t - jk * st;
            C<R> acc = C<R>{(R)0, (R)0};
            for (int q = 0; q < CHI; ++q) acc = cfma(cur[base + q * st], Xs[k * CC + q * CHI + jk], acc);
            nxt[t] = acc;
        }
        __syncthreads();
        C<R>* tmp = cur;
        cur = nxt;
        nxt = tmp;
    }
    C<R>* g = (C<R>*)a.Gamma + (size_t)v * H2;
    for (int t = threadIdx.x; t < H2; t += blockDim.x) g[t] = cur[t];
}

// rho_a = sum_J Gamma[i, J] conj(Gamma[i', J]) prod_k lambda_k[j_k]^2 / trace (Eqs. (partial_dens),
// (bp_approx)); read-out +1 if rho_a[0][0] > 1/2 (Eq. (rounding_rule)).  One warp per vertex.
template <int CHI, int D, typename R>
__global__ void plain_marginals_kernel(const C<R>* Gamma, const double* lam, const int4* vslots, int n, cd* rho,
                                       int8_t* sign, int* nan_flag) {
    constexpr int H = PlainShape<CHI, D, R>::H;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (warp >= n) return;
    const int v = warp;
    const int4 sl = vslots[v];
    cd acc[4] = {cd{0, 0}, cd{0, 0}, cd{0, 0}, cd{0, 0}};
    for (int r = lane; r < H; r += 32) {
        int rem = r;
        double wgt = 1.0;
        for (int k = D - 1; k >= 0; --k) {
            const double l = lam_get(lam, CHI, plain_slot_edge(sl, k), rem % CHI);
            wgt *= l * l;
            rem /= CHI;
        }
        const cd g0 = ccast<double>(Gamma[(size_t)v * 2 * H + r]), g1 = ccast<double>(Gamma[(size_t)v * 2 * H + H + r]);
        acc[0] = cfmac(g0, wgt * g0, acc[0]);
        acc[1] = cfmac(g1, wgt * g0, acc[1]);
        acc[2] = cfmac(g0, wgt * g1, acc[2]);
        acc[3] = cfmac(g1, wgt * g1, acc[3]);
    }
    for (int q = 0; q < 4; ++q) {
        acc[q].x = group_sum<32>(acc[q].x, 0xffffffffu);
        acc[q].y = group_sum<32>(acc[q].y, 0xffffffffu);
    }
    if (lane == 0) {
        const double tr = acc[0].x + acc[3].x;
        const double it = 1.0 / tr;
        for (int q = 0; q < 4; ++q) rho[(size_t)v * 4 + q] = it * acc[q];
        if (sign) sign[v] = (acc[0].x * it > 0.5) ? 1 : -1;
        if (!(tr == tr) || tr == 0.0) atomicOr(nan_flag, 1);
    }
}

// Residual R of the local-orthogonality condition (App. C) on the plain layout: one block of
// max(CHI^2/2, 1) threads per (vertex, slot) item whose slot holds a bond,
//   D_k[j, j'] = delta_{j j'} [lambda_k[j] > 0] - sum_{i, J \ j_k} Gamma[i, J(j)] conj(Gamma[i, J(j')])
//                prod_{l != k} lambda_l[j_l]^2
// in FP64 (complex64 Gamma is widened), then its trace norm (FP64 one-sided Jacobi), added to
// *out.  The caller divides the sum by 2|E|.
template <int CHI, int D, typename R>
__global__ void plain_residual_kernel(const C<R>* Gamma, const double* lam, const int4* vslots, double* out) {
    constexpr int H = PlainShape<CHI, D, R>::H, CC = CHI * CHI, NO = H / CHI;
    __shared__ cd A[CC];
    __shared__ double tn;
    __shared__ int flag;
    const int v = blockIdx.x / D, k = blockIdx.x % D;
    const int4 sl = vslots[v];
    const int ek = plain_slot_edge(sl, k);
    if (ek < 0) return;   // a phantom slot: the whole block leaves
    const int g = threadIdx.x;
    const C<R>* gv = Gamma + (size_t)v * 2 * H;
    int sk = 1;   // stride of slot k, CHI^(D-1-k)
    for (int l = D - 1; l > k; --l) sk *= CHI;
    for (int r = g; r < CC; r += blockDim.x) {
        const int j = r / CHI, jp = r % CHI;
        cd acc = cd{0.0, 0.0};
        for (int q = 0; q < NO; ++q) {
            // q runs over the indices of the other slots (last slot fastest)
            int rem = q, base = 0, stride = 1;
            double w = 1.0;
            for (int l = D - 1; l >= 0; --l) {
                if (l != k) {
                    const int idx = rem % CHI;
                    rem /= CHI;
                    const double lv = lam_get(lam, CHI, plain_slot_edge(sl, l), idx);
                    w *= lv * lv;
                    base += idx * stride;
                }
                stride *= CHI;
            }
            for (int i = 0; i < 2; ++i) {
                const cd x = ccast<double>(gv[i * H + base + j * sk]), y = ccast<double>(gv[i * H + base + jp * sk]);
                acc = cfmac(y, w * x, acc);
            }
        }
        const double act = (j == jp && lam_get(lam, CHI, ek, j) > 0.0) ? 1.0 : 0.0;
        A[r] = cd{act - acc.x, -acc.y};
    }
    if (g == 0) tn = 0.0;
    __syncthreads();
    BlockGroup grp{&flag};
    jacobi_svd<CHI, double, BlockGroup, false>(A, nullptr, g, grp, group_mask<CHI>(), 1e-15, 60, false);
    __syncthreads();
    if (g < CHI) {
        double c2 = 0.0;
        for (int r = 0; r < CHI; ++r) c2 += norm2(A[g * CHI + r]);
        atomicAdd(&tn, sqrt(c2));
    }
    __syncthreads();
    if (g == 0) atomicAdd(out, tn);
}

// One step of the measurement sampling of Sec. IV A on the plain layout (one warp, vertex a):
// p0 = rho_a[0][0] as in plain_marginals_kernel, the outcome x_a = +1 if u < p0 (else -1) and its
// probability, then the projection of Eq. (projection): the other physical component of
// Gamma_a is zeroed.
template <int CHI, int D, typename R>
__global__ void plain_sample_kernel(C<R>* Gamma, const double* lam, const int4* vslots, int a, double u, int step,
                                    int8_t* x_out, double* p_out) {
    constexpr int H = PlainShape<CHI, D, R>::H;
    const int lane = threadIdx.x & 31;
    const int4 sl = vslots[a];
    C<R>* g = Gamma + (size_t)a * 2 * H;
    double r00 = 0.0, r11 = 0.0;
    for (int r = lane; r < H; r += 32) {
        int rem = r;
        double wgt = 1.0;
        for (int k = D - 1; k >= 0; --k) {
            const double l = lam_get(lam, CHI, plain_slot_edge(sl, k), rem % CHI);
            wgt *= l * l;
            rem /= CHI;
        }
        r00 += wgt * norm2(ccast<double>(g[r]));
        r11 += wgt * norm2(ccast<double>(g[H + r]));
    }
    r00 = group_sum<32>(r00, 0xffffffffu);
    r11 = group_sum<32>(r11, 0xffffffffu);
    const double p0 = r00 / (r00 + r11);
    const int keep = u < p0 ? 0 : 1;
    if (lane == 0) {
        x_out[a] = keep == 0 ? 1 : -1;
        p_out[step] = keep == 0 ? p0 : r11 / (r00 + r11);
    }
    for (int r = lane; r < H; r += 32) g[(1 - keep) * H + r] = C<R>{(R)0, (R)0};
}

// ---------------------------------------------------------------------------
// The simple update of a diagonal gate (App. E) in QR-reduced form, as on the persistent path: each
// side and physical index is one block A_{x,i}[J, j] = w_x[J] Gamma_x[i][j][J] (CHI^(D-1) x CHI),
//   M[(i_a r), (i_b r')] = ph(i_a, i_b) sum_j R_{a,i_a}[r, j] lambda_j R_{b,i_b}[r', j]
// (2 CHI x 2 CHI) has the singular values of Theta, and the new tensors come from the reflectors.
// One block of threads per edge, one launch per colour.  Against the whole-side update of
// gtqa_general.cuh, which takes any 4 x 4 gate, the core has half the order, so an eighth of the
// SVD work.  The last gate of a vertex in the layer applies the mixing gate exp(-i t_X X) to it,
// the first one the leading mixing gate.
// ---------------------------------------------------------------------------
struct PlainGateArgs {
    void* Gamma;
    double* lam;
    const int4* edge_info;
    const int4* vslots;
    const int* gate_edge;     // edges of this launch
    const int* gate_bits;     // first gate of u, of v; last gate of u, of v
    int count;
    const double* J;
    const double* hd;         // h_a / degree of a
    double* stats;
    Control* ctl;
    int chi;
    double svd_cut;
    double tZ, cX, sX;        // mixing gate after a vertex's last gate
    int pre;                  // leading mixing gate before its first one
    double cXp, sXp;
    void* scratch;            // CHI = 16: reflectors, [gates in launch][4][CHI^2][CHI]
};

// The four diagonal gate phases of edge e: lane d = 2 i_a + i_b < 4.
__device__ __forceinline__ cd ising_phase(double tZ, double J, double ha, double hb, int d) {
    const double za = 1.0 - 2.0 * (d >> 1), zb = 1.0 - 2.0 * (d & 1);
    double sn, cs;
    sincos(-tZ * (J * za * zb + ha * za + hb * zb), &sn, &cs);
    return cd{cs, sn};
}
// [[c, -i s], [-i s, c]] on the pair (g0, g1)
template <typename TS>
__device__ __forceinline__ void mix_pair(C<TS>& g0, C<TS>& g1, double c, double s) {
    const cd a0 = ccast<double>(g0), a1 = ccast<double>(g1);
    g0 = ccast<TS>(cd{c * a0.x + s * a1.y, c * a0.y - s * a1.x});
    g1 = ccast<TS>(cd{s * a0.y + c * a1.x, -s * a0.x + c * a1.y});
}

template <int CHI, int D>
struct PlainGateShape {
    static constexpr int NR = ipow(CHI, D - 1), G = NR / 2, TEAM = 4 * G, NM = 2 * CHI, LS = NM * NM / 2;
    static_assert(G <= 32 && LS <= TEAM, "one warp per block at most");
};

template <int CHI, int D, typename TS, typename R>
struct PlainGateSm {
    using S = PlainGateShape<CHI, D>;
    C<R> U[4][CHI][S::NR];     // scaled reflectors, then the new tensors
    C<R> M[S::NM * S::NM];
    C<R> V[S::NM * S::NM];     // first the R factors [block][row][col]
    C<R> T[sizeof(R) == 8 ? S::NM * S::NM : 1];
    cf M32[sizeof(R) == 8 ? S::NM * S::NM : 1];
    cf V32[sizeof(R) == 8 ? S::NM * S::NM : 1];
    double lab[CHI];
    double n2[S::NM], isig[CHI];
    C<R> ph[4];
    int perm[S::NM];
    int keep, flag, nrot;
    unsigned relmask;
};

template <int CHI, int D, typename TS, typename R>
__global__ void __launch_bounds__(PlainGateShape<CHI, D>::TEAM) plain_ising_kernel(PlainGateArgs c) {
    using S = PlainGateShape<CHI, D>;
    using CR = C<R>;
    using CT = C<TS>;
    constexpr int NM = S::NM, NR = S::NR, G = S::G, TEAM = S::TEAM, LS = S::LS, H = ipow(CHI, D);
    extern __shared__ __align__(16) unsigned char plain_smem[];
    PlainGateSm<CHI, D, TS, R>& sm = *reinterpret_cast<PlainGateSm<CHI, D, TS, R>*>(plain_smem);
    auto bar = [&]() {
        if constexpr (TEAM < 32) __syncwarp(group_mask<TEAM>());
        else __syncthreads();
    };
    const int tid = threadIdx.x, blk = tid / G, l = tid % G, x = blk >> 1, i = blk & 1;
    const unsigned gm = group_mask<G>();
    const int e = c.gate_edge[blockIdx.x], bits = c.gate_bits[blockIdx.x];
    const int4 ei = c.edge_info[e];
    const int slot2[2] = {ei.z, ei.w}, vtx2[2] = {ei.x, ei.y};
    // offset of row J (the other slots, last one fastest) inside a vertex tensor, side x
    auto row_off = [&](int slot, int J) {
        int off = 0;
        for (int k = D - 1; k >= 0; --k)
            if (k != slot) {
                off += (J % CHI) * ipow(CHI, D - 1 - k);
                J /= CHI;
            }
        return off;
    };
    CT* Gam = (CT*)c.Gamma;
    CR y0[CHI], y1[CHI];
    double w0 = 1.0, w1 = 1.0;
    {
        const int slot = slot2[x], ss = ipow(CHI, D - 1 - slot);
        const int4 sl = c.vslots[vtx2[x]];
        const int es[4] = {sl.x, sl.y, sl.z, sl.w};
        int J0 = l, J1 = l + G;
        for (int k = D - 1; k >= 0; --k)
            if (k != slot) {
                w0 *= lam_get(c.lam, CHI, es[k], J0 % CHI);
                w1 *= lam_get(c.lam, CHI, es[k], J1 % CHI);
                J0 /= CHI;
                J1 /= CHI;
            }
        const CT* g = Gam + (size_t)vtx2[x] * 2 * H;
        const int f0 = row_off(slot, l), f1 = row_off(slot, l + G);
        const bool lead = c.pre && ((bits >> x) & 1);
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) {
            CT a = g[i * H + f0 + cc * ss], b = g[i * H + f1 + cc * ss];
            if (lead) {   // own component of the mixed pair; mix_pair is symmetric in the two
                CT a2 = g[(i ^ 1) * H + f0 + cc * ss], b2 = g[(i ^ 1) * H + f1 + cc * ss];
                mix_pair(a, a2, c.cXp, c.sXp);
                mix_pair(b, b2, c.cXp, c.sXp);
            }
            y0[cc] = (R)w0 * ccast<R>(a);
            y1[cc] = (R)w1 * ccast<R>(b);
        }
        if (tid < CHI) sm.lab[tid] = c.lam[(size_t)e * CHI + tid];
        if (tid < 4) sm.ph[tid] = ccast<R>(ising_phase(c.tZ, c.J[e], c.hd[ei.x], c.hd[ei.y], tid));
        if (tid == 0) sm.nrot = 0;
        bar();
    }
    qr_steps<CHI, G, 0>(y0, y1, &sm.U[blk][0][0], l, gm);
    // rows l and, where the group is smaller than CHI, l + G of R
#pragma unroll
    for (int cc = 0; cc < CHI; ++cc) {
        const R lb = x == 0 ? (R)sm.lab[cc] : (R)1;
        if (l < CHI && cc >= l) sm.V[(blk * CHI + l) * CHI + cc] = lb * y0[cc];
    }
    bar();
    for (int t = tid; t < NM * NM; t += TEAM) {
        const int col = t / NM, row = t % NM;
        const int ia = row / CHI, r = row % CHI, ib = col / CHI, rp = col % CHI;
        const CR* Ra = sm.V + (ia * CHI + r) * CHI;
        const CR* Rb = sm.V + ((2 + ib) * CHI + rp) * CHI;
        CR acc = CR{(R)0, (R)0};
        for (int j = r > rp ? r : rp; j < CHI; ++j) acc = cfma(Ra[j], Rb[j], acc);
        sm.M[t] = sm.ph[2 * ia + ib] * acc;
    }
    bar();
    if (tid < LS) {
        SvdCount done;
        auto run = [&](const auto& grp) {
            done = core_svd<NM>(sm.M, sm.V, sm.M32, sm.V32, sm.T, sm.n2, &sm.relmask, tid, grp, c.svd_cut, c.chi);
            if (done.rot) atomicAdd(&sm.nrot, done.rot);
            if (tid < NM) sm.perm[desc_rank_bits(sm.n2, NM, tid)] = tid;
            grp.sync();
        };
        if constexpr (LS <= 32) run(WarpGroup{group_mask<LS>()});
        else run(TeamGroup<LS>{0, &sm.flag});
        if (tid < NM) {
            const int k = truncate_core<NM, CHI, false>(sm.n2, sm.perm, sm.isig, c.lam + (size_t)e * CHI, c.stats, c.chi,
                                                        c.svd_cut, tid);
            if (tid == 0) {
                atomicAdd(&c.stats[2], (double)done.pairs);
                atomicAdd(&c.stats[3], (double)sm.nrot);
                sm.keep = k;
            }
        }
    }
    bar();
    const int keep = sm.keep;
    CR E0[CHI], E1[CHI];
#pragma unroll
    for (int cc = 0; cc < CHI; ++cc) {
        E0[cc] = E1[cc] = CR{(R)0, (R)0};
        if (l < CHI && cc < keep) {
            const int pc = sm.perm[cc], row = i * CHI + l;
            E0[cc] = x == 0 ? (R)sm.isig[cc] * sm.M[pc * NM + row] : conj(sm.V[pc * NM + row]);
        }
    }
    apply_reflectors<CHI, G>(E0, E1, &sm.U[blk][0][0], l, gm);
    const R iw0 = w0 > 0.0 ? (R)nr_rcp(w0) : (R)0, iw1 = w1 > 0.0 ? (R)nr_rcp(w1) : (R)0;
    bar();   // everyone is done reading the reflectors
#pragma unroll
    for (int cc = 0; cc < CHI; ++cc) {
        sm.U[blk][cc][l] = iw0 * E0[cc];
        sm.U[blk][cc][l + G] = iw1 * E1[cc];
    }
    bar();
    for (int t = tid; t < 2 * CHI * NR; t += TEAM) {
        const int xx = t / (CHI * NR), rem = t % (CHI * NR), col = rem / NR, row = rem % NR;
        CT g0 = ccast<TS>(sm.U[2 * xx][col][row]), g1 = ccast<TS>(sm.U[2 * xx + 1][col][row]);
        if ((bits >> (2 + xx)) & 1) mix_pair(g0, g1, c.cX, c.sX);
        CT* g = Gam + (size_t)vtx2[xx] * 2 * H + row_off(slot2[xx], row) + col * ipow(CHI, D - 1 - slot2[xx]);
        g[0] = g0;
        g[H] = g1;
    }
}

// exp(-i t X) on the vertices of a list (those without edges)
template <int CHI, int D, typename TS>
__global__ void plain_mixing_kernel(void* Gamma, const int* vertex, double c, double s) {
    constexpr int H = ipow(CHI, D);
    C<TS>* g = (C<TS>*)Gamma + (size_t)vertex[blockIdx.x] * 2 * H;
    for (int r = threadIdx.x; r < H; r += blockDim.x) {
        C<TS> g0 = g[r], g1 = g[H + r];
        mix_pair(g0, g1, c, s);
        g[r] = g0;
        g[H + r] = g1;
    }
}

// ---------------------------------------------------------------------------
// CHI = 16, degree 3: the same update, one block of 512 threads per edge.
//
// What bounds it: the FP64 pipe.  The useful products of one gate are, per block of
// CHI^2 x CHI, 30k complex products each for the QR's inner products, its updates and the
// reflectors' Gram matrix, and 64k for the back-application.  So:
//  * one side at a time, 256 lanes per block of it, each with its row of 16 columns in registers
//    (the panel of both sides, 256 KB in FP64, fits neither shared memory nor the registers);
//    finished reflectors go to global scratch once and are read back once;
//  * the inner products of a step with all other columns (later ones for the QR, earlier ones for
//    the Gram matrix of the reflectors) are summed together, 31 values by one reduce-scatter per
//    warp; the scalars of a step are formed by one warp of the block, not by all;
//  * the back-application is one product E - U Z per row with Z from (I + strict upper(U^H U)) Z =
//    U^H E (compact WY form), instead of 16 reductions over 256 rows;
//  * columns beyond the bond's current dimension (lambda = 0) are skipped, and the core is
//    decomposed at the order (8, 16 or 32) that holds both of its halves.
// ---------------------------------------------------------------------------
template <typename R>
struct Gate16Sm {
    using CR = C<R>;
    static constexpr int CHI = 16, NM = 32, NR = 256;
    CR M[NM * NM];
    CR V[NM * NM];            // first the R factors [block][row][col]
    CR T[NM * NM];            // scratch of the SVD; then Z [block][j][col]
    cf M32[sizeof(R) == 8 ? NM * NM : 1];
    cf V32[sizeof(R) == 8 ? NM * NM : 1];
    CR SU[4][CHI][CHI];       // u_j^H u_k, j < k
    CR top[4][CHI][CHI];      // rows 0 .. 15 of the reflectors, [block][k][row]
    R red[2][8][32];          // partial sums, [block of the side][warp][value]
    CR wv[2][CHI];            // tau v^H y of the later columns
    R st[2];
    CR vkk[2];
    double lab[CHI];
    double n2[NM], isig[CHI];
    CR ph[4];
    int perm[NM];
    int keep, flag, nrot;
    unsigned relmask;
};

// Step K of the QR of the two blocks of one side: lane `row` of block i holds y[0 .. 15].  nc: the
// columns in use.  vd: this row's diagonal reflector entry (row < CHI).
template <int K, typename R>
__device__ __forceinline__ void qr16_steps(C<R> (&y)[16], C<R>& vd, Gate16Sm<R>& sm, C<R>* U, int blk, int i, int row,
                                           int nc) {
    if constexpr (K < 16) {
        using CR = C<R>;
        if (K >= nc) return;
        const int lane = threadIdx.x & 31, warp = row / 32;
        const CR z = CR{(R)0, (R)0};
        const CR x = row >= K ? y[K] : z;
        // |x|^2 and the inner products of x with the 15 other columns, in two groups of 16 values
        // (registers); value v of a group ends on lane 2 v
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            R s[16];
            s[0] = half == 0 ? norm2(x) : (R)0;
            s[15] = (R)0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int c = half == 0 ? q - 1 : 7 + q;   // other column, skipping K
                if (c < 0) continue;
                const int col = c < K ? c : c + 1, at = half == 0 ? 2 * q - 1 : 2 * q;
                CR d = z;
                if (col < nc) {
                    // an earlier column: its reflector, below the diagonal and vd on it
                    const CR a = c < K ? (row > c ? y[c] : (row == c ? vd : z)) : y[col];
                    d = c < K ? cfmac(a, x, z) : cfmac(x, a, z);
                }
                s[at] = d.x;
                s[at + 1] = d.y;
            }
            rs_level<16, 16>(s, 0xffffffffu, lane);
            if ((lane & 1) == 0) sm.red[i][warp][16 * half + lane / 2] = s[0];
        }
        __syncthreads();
        if (warp == 0) {
            // value v on lane v
            R t = (R)0;
#pragma unroll
            for (int w = 0; w < 8; ++w) t += sm.red[i][w][lane];
            const R x2 = __shfl_sync(0xffffffffu, t, 0);
            const CR xkk = CR{__shfl_sync(0xffffffffu, y[K].x, K), __shfl_sync(0xffffffffu, y[K].y, K)};
            const R a2 = norm2(xkk);
            const R arg = (lane & 1) ? a2 : x2;
            const R rs = arg > tiny_norm2<R>() ? nr_rsqrt(arg) : (R)0;
            const R r0 = __shfl_sync(0xffffffffu, rs, 0), ra = __shfl_sync(0xffffffffu, rs, 1);
            const R nrm = x2 * r0, axkk = a2 * ra;
            const CR ph = nonzero(ra) ? CR{xkk.x * ra, xkk.y * ra} : CR{(R)1, (R)0};
            const R stau = nonzero(nrm) ? nr_rsqrt(nrm * (nrm + axkk)) : (R)0;
            const CR pv = nrm * ph;
            // lane c < 15: the sum of column c (earlier) or c + 1 (later), and row K of that column
            const int at = lane < 7 ? 1 + 2 * lane : 2 + 2 * (lane % 15);
            const CR sum = CR{__shfl_sync(0xffffffffu, t, at), __shfl_sync(0xffffffffu, t, at + 1)};
            CR yk = z;
#pragma unroll
            for (int c = 0; c < 15; ++c) {
                const CR a = y[c < K ? c : c + 1];
                const R bx = __shfl_sync(0xffffffffu, a.x, K), by = __shfl_sync(0xffffffffu, a.y, K);
                if (lane == c) yk = CR{bx, by};
            }
            if (lane < K) {
                // v_c^H v_K = v_c^H x + conj(v_c[K]) pv, scaled to u
                const CR g = cfmac(yk, pv, sum);
                sm.SU[blk][lane][K] = (stau * sm.SU[blk][lane][lane].x) * g;
            } else if (lane < 15) {
                sm.wv[i][lane + 1] = (stau * stau) * cfmac(pv, yk, sum);   // tau (x^H y + conj(pv) y_K)
            }
            if (lane == K) {
                sm.SU[blk][K][K] = CR{stau, (R)0};   // kept for the scaling of later columns
                sm.st[i] = stau;
                sm.vkk[i] = xkk + pv;
                y[K] = CR{-pv.x, -pv.y};
                vd = xkk + pv;
            }
        }
        __syncthreads();
        const R stau = sm.st[i];
        const CR v = row == K ? sm.vkk[i] : x;
#pragma unroll
        for (int c = K + 1; c < 16; ++c)
            if (c < nc && row >= K) y[c] = cfms(v, sm.wv[i][c], y[c]);
        const CR u = stau * v;
        U[K * 256 + row] = u;
        if (row < 16) sm.top[blk][K][row] = u;
        qr16_steps<K + 1>(y, vd, sm, U, blk, i, row, nc);
    }
}

template <typename TS, typename R>
__global__ void __launch_bounds__(512, 1) ising16_gate_kernel(PlainGateArgs c) {
    using CR = C<R>;
    using CT = C<TS>;
    constexpr int CHI = 16, NR = 256, H = CHI * CHI * CHI;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    Gate16Sm<R>& sm = *reinterpret_cast<Gate16Sm<R>*>(plain_smem);
    const int tid = threadIdx.x, i = tid / NR, row = tid % NR;
    const int e = c.gate_edge[blockIdx.x], bits = c.gate_bits[blockIdx.x];
    const int4 ei = c.edge_info[e];
    CT* Gam = (CT*)c.Gamma;
    CR* Us = reinterpret_cast<CR*>(c.scratch) + (size_t)blockIdx.x * 4 * CHI * NR;   // [blk][k][row]
    if (tid < CHI) sm.lab[tid] = c.lam[(size_t)e * CHI + tid];
    if (tid >= 32 && tid < 36) sm.ph[tid - 32] = ccast<R>(ising_phase(c.tZ, c.J[e], c.hd[ei.x], c.hd[ei.y], tid - 32));
    if (tid == 0) sm.nrot = 0;
    __syncthreads();
    int nc = 0;   // the bond's current dimension
    for (int j = 0; j < CHI; ++j) nc = sm.lab[j] > 0.0 ? j + 1 : nc;
    nc = nc > 0 ? nc : 1;
    double w2[2];
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int slot = x ? ei.w : ei.z, vtx = x ? ei.y : ei.x, blk = 2 * x + i;
        const int4 ve = c.vslots[vtx];
        int o0, o1;
        others_of(slot, o0, o1);
        const int e0 = plain_slot_edge(ve, o0), e1 = plain_slot_edge(ve, o1);
        const double w = lam_get(c.lam, CHI, e0, row / CHI) * lam_get(c.lam, CHI, e1, row % CHI);
        if (x == 0) w2[0] = w;
        else w2[1] = w;
        auto stride = [](int k) { return k == 0 ? CHI * CHI : (k == 1 ? CHI : 1); };
        const int ss = stride(slot);
        const CT* g = Gam + (size_t)vtx * 2 * H + row / CHI * stride(o0) + row % CHI * stride(o1);
        const bool lead = c.pre && ((bits >> x) & 1);
        CR y[CHI];
        CR vd = CR{(R)0, (R)0};
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) {
            CT a = g[i * H + cc * ss];
            if (lead) {
                CT b = g[(i ^ 1) * H + cc * ss];
                mix_pair(a, b, c.cXp, c.sXp);
            }
            y[cc] = (R)w * ccast<R>(a);
        }
        qr16_steps<0>(y, vd, sm, Us + (size_t)blk * CHI * NR, blk, i, row, nc);
        if (row < CHI) {
#pragma unroll
            for (int cc = 0; cc < CHI; ++cc)
                if (cc >= row) sm.V[(blk * CHI + row) * CHI + cc] = x == 0 ? (R)sm.lab[cc] * y[cc] : y[cc];
        }
        __syncthreads();
    }
    // ---- core with the diagonal gate at order 2 hc, column-major ----
    const int hc = nc <= 4 ? 4 : (nc <= 8 ? 8 : 16), NM = 2 * hc;
    for (int t = tid; t < NM * NM; t += 512) {
        const int col = t / NM, rw = t % NM;
        const int ia = rw / hc, r = rw % hc, ib = col / hc, rp = col % hc;
        const CR* Ra = sm.V + (ia * CHI + r) * CHI;
        const CR* Rb = sm.V + ((2 + ib) * CHI + rp) * CHI;
        CR acc = CR{(R)0, (R)0};
        for (int j = r > rp ? r : rp; j < nc; ++j) acc = cfma(Ra[j], Rb[j], acc);
        sm.M[t] = sm.ph[2 * ia + ib] * acc;
    }
    __syncthreads();
    auto solve = [&](auto order, const auto& grp) {
        constexpr int N = decltype(order)::value;
        SvdCount done = core_svd<N>(sm.M, sm.V, sm.M32, sm.V32, sm.T, sm.n2, &sm.relmask, tid, grp, c.svd_cut, c.chi);
        if (done.rot) atomicAdd(&sm.nrot, done.rot);
        if (tid < N) sm.perm[desc_rank_bits(sm.n2, N, tid)] = tid;
        grp.sync();
        if (tid < N) {
            const int k = truncate_core<N, (N < CHI ? N : CHI), false>(sm.n2, sm.perm, sm.isig, c.lam + (size_t)e * CHI, c.stats,
                                                                       c.chi, c.svd_cut, tid);
            if (tid == 0) {
                atomicAdd(&c.stats[2], (double)done.pairs);
                atomicAdd(&c.stats[3], (double)sm.nrot);
                sm.keep = k;
            }
        }
        // a core of order 8 has no more than 8 triplets; the bond's other weights are zero
        if (N < CHI && tid < CHI - N) c.lam[(size_t)e * CHI + N + tid] = 0.0;
    };
    if (hc == 4) {
        if (tid < 32) solve(std::integral_constant<int, 8>{}, WarpGroup{0xffffffffu});
    } else if (hc == 8) {
        if (tid < 128) solve(std::integral_constant<int, 16>{}, TeamGroup<128>{0, &sm.flag});
    } else {
        solve(std::integral_constant<int, 32>{}, BlockGroup{&sm.flag});
    }
    __syncthreads();
    const int keep = sm.keep;
    // ---- Z of every block: Y = U^H E (E has its first nc rows only), then back substitution ----
    auto etop = [&](int blk, int r, int cc) {   // row r < nc of column cc < keep
        const int pc = sm.perm[cc], rw = (blk & 1) * hc + r;
        return blk < 2 ? (R)sm.isig[cc] * sm.M[pc * NM + rw] : conj(sm.V[pc * NM + rw]);
    };
    for (int t = tid; t < 4 * CHI * CHI; t += 512) {
        const int blk = t / (CHI * CHI), j = (t / CHI) % CHI, cc = t % CHI;
        CR acc = CR{(R)0, (R)0};
        if (j < nc && cc < keep)
            for (int r = j; r < nc; ++r) acc = cfmac(sm.top[blk][j][r], etop(blk, r, cc), acc);
        sm.T[t] = acc;
    }
    __syncthreads();
    if (tid % 128 < CHI) {   // one lane per column, the blocks on different warps
        const int blk = tid / 128, cc = tid % 128;
        if (cc < keep) {
            CR* Z = sm.T + blk * CHI * CHI + cc;
            for (int j = nc - 2; j >= 0; --j) {
                CR acc = Z[j * CHI];
                for (int k = j + 1; k < nc; ++k) acc = cfms(sm.SU[blk][j][k], Z[k * CHI], acc);
                Z[j * CHI] = acc;
            }
        }
    }
    __syncthreads();
    // ---- new tensors, row by row ----
#pragma unroll 1
    for (int x = 0; x < 2; ++x) {
        const int slot = x ? ei.w : ei.z, vtx = x ? ei.y : ei.x, blk = 2 * x + i;
        int o0, o1;
        others_of(slot, o0, o1);
        CR E[CHI];
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) E[cc] = row < nc && cc < keep ? etop(blk, row, cc) : CR{(R)0, (R)0};
        const CR* Ub = Us + (size_t)blk * CHI * NR + row;
        for (int j = 0; j < nc; ++j) {
            const CR u = Ub[j * NR];
            const CR* Z = sm.T + (blk * CHI + j) * CHI;
#pragma unroll
            for (int cc = 0; cc < CHI; ++cc)
                if (cc < keep) E[cc] = cfms(u, Z[cc], E[cc]);
        }
        const double w = x ? w2[1] : w2[0];
        const R iw = w > 0.0 ? (R)nr_rcp(w) : (R)0;
        auto stride = [](int k) { return k == 0 ? CHI * CHI : (k == 1 ? CHI : 1); };
        const int ss = stride(slot);
        CT* gv = Gam + (size_t)vtx * 2 * H;
        CT* g = gv + (size_t)i * H + row / CHI * stride(o0) + row % CHI * stride(o1);
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) g[cc * ss] = ccast<TS>(iw * E[cc]);
        if ((bits >> (2 + x)) & 1) {   // the mixing gate after the vertex's last gate
            __syncthreads();
            for (int r = tid; r < H; r += 512) {
                CT g0 = gv[r], g1 = gv[H + r];
                mix_pair(g0, g1, c.cX, c.sX);
                gv[r] = g0;
                gv[H + r] = g1;
            }
        }
    }
}

}  // namespace gtqa
