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
//            diag(lambda)/sum(lambda) (Eq. (reconstructed_messages)); then one cooperative launch
//            runs the flooding sweeps of Eq. (local_consistency) and their stopping rule (App. B);
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
    void* msg[2];             // the message buffers; ctl->cur is the current one
    void* X;                  // regauge transforms [m][2][CHI^2]
    void* dm;                 // [2m][CHI^2]: new - old of every message of a sweep
    const int4* vslots;       // slots per vertex (x, y, z, w; -1 phantom)
    const int4* edge_info;    // (u, v, slot at u, slot at v)
    int n, m;
    int warm;
    void* D0;                 // mixed mode: [2m][CHI^2] warm-start defect F(m0) - tr F(m0) m0 (storage type)
    cd* t0;                   // mixed mode: [2m] tr F(m0)
    Control* ctl;
};

template <int CHI, int D, typename R, typename RC = R>
struct PlainShape {
    static constexpr int H = ipow(CHI, D), H2 = 2 * H, CC = CHI * CHI;
    static constexpr bool MIX = sizeof(R) != sizeof(RC);
    // team of one (vertex, physical index) item, and the outputs of a fiber per lane
    static constexpr int NT = CHI == 16 ? 512 : (CHI == 8 || (D == 4 && CHI == 4) ? 128 : (CHI == 4 ? 64 : 32));
    static constexpr int XO = H > NT ? H / NT : 1;
    static constexpr int ITEMS = H / XO, PARTS = NT / CC;
    static constexpr int TPB = 512, TEAMS = TPB / NT;
    static constexpr int PH = H + H / CC;                // one padding element per CHI^2 plane
    static constexpr int NB = D == 4 ? 4 : 3;            // T, prefix, suffix (and one more)
    static constexpr bool RANK = CHI >= 8;               // skip indices beyond the bonds' dimensions
    static constexpr size_t team_smem = sizeof(C<R>) * (NB * PH + (MIX ? 2 : 1) * D * CC) + sizeof(R) * D * CHI +
                                        sizeof(int) * 16;
    static constexpr int GL = CC / 2 > 1 ? CC / 2 : 1;   // lanes of a trace norm
    static constexpr int GROUPS = TPB / GL < 64 ? TPB / GL : 64;
    static constexpr size_t group_smem =
        sizeof(RC) == 8 ? (size_t)CC * (3 * sizeof(cd) + 2 * sizeof(cf)) + 2 * CHI * sizeof(double) : (size_t)CC * sizeof(cf) + 16;
    static constexpr size_t bp_smem = (TEAMS * ((team_smem + 15) / 16 * 16) > GROUPS * ((group_smem + 15) / 16 * 16)
                                           ? TEAMS * ((team_smem + 15) / 16 * 16)
                                           : GROUPS * ((group_smem + 15) / 16 * 16));
    static constexpr size_t init_smem = MIX ? sizeof(cd) * (H2 + H2 / CC) : 0;
    static constexpr size_t vertex_smem = sizeof(C<R>) * (PH + CC);
};

// Whether an earlier launch on this state failed (a NaN distance, a barrier that gave up).  The host reads
// the status once per call, so the BP runs and regauges behind a failed launch leave by themselves: a
// barrier that gave up leaves a count that is no multiple of the grid, and messages half written.  The
// load is issued at a kernel's start and used where it waits or writes first, so that it costs no latency.
__device__ __forceinline__ bool run_failed(const Control* ctl) { return __ldcg(&ctl->err) != 0; }

__device__ __forceinline__ int plain_slot_edge(const int4& v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}

// T = Gamma prod_k lambda_k^{1/2}; with warm, the vertex's outgoing messages are set to
// diag(lambda)/sum(lambda) (mixed: delta = 0) in the current message buffer.  One block per vertex.
// Mixed: F0 = F(m0) of every outgoing message in FP64 from the stored T (so that F(m0 + delta) =
// F0 + F_delta holds for the T that the sweeps contract), kept as D0 = F0 - tr(F0) m0 and t0.  As on
// the persistent path the weights are folded into T~ = T prod m0^{1/2} once, so that a term is one
// complex product (4 FP64 instructions instead of 12), and only j <= j' is summed.
template <int CHI, int D, typename R, typename RC = R>
__global__ void __launch_bounds__(256) plain_bp_init_kernel(PlainArgs a) {
    using S = PlainShape<CHI, D, R, RC>;
    constexpr bool MIX = S::MIX;
    constexpr int CC = S::CC, H = S::H, H2 = S::H2;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    const int v = blockIdx.x;
    __shared__ RC sq[D][CHI], m0[D][CHI], rt[D][CHI];
    const int4 sl = a.vslots[v];
    if (threadIdx.x < D * CHI) {
        const int k = threadIdx.x / CHI, j = threadIdx.x % CHI;
        const int e = plain_slot_edge(sl, k);
        const RC lj = lam_get(a.lam, CHI, e, j);
        sq[k][j] = sqrt(lj);
        RC s = 0.0;
        for (int q = 0; q < CHI; ++q) s += lam_get(a.lam, CHI, e, q);
        m0[k][j] = s > 0.0 ? lj / s : 0.0;
        if constexpr (MIX) rt[k][j] = s > 0.0 ? sqrt(lj / s) : 0.0;
    }
    __syncthreads();
    const C<R>* g = (const C<R>*)a.Gamma + (size_t)v * H2;
    C<R>* T = (C<R>*)a.T + (size_t)v * H2;
    cd* Tm = reinterpret_cast<cd*>(plain_smem);
    for (int t = threadIdx.x; t < H2; t += blockDim.x) {
        int r = t % H;
        RC f = 1.0, w = 1.0;
#pragma unroll
        for (int k = D - 1; k >= 0; --k) {
            f *= sq[k][r % CHI];
            if constexpr (MIX) w *= rt[k][r % CHI];
            r /= CHI;
        }
        const C<R> tv = ccast<R>(f * ccast<RC>(g[t]));
        T[t] = tv;
        if constexpr (MIX) Tm[t + t / CC] = w * ccast<double>(tv);
    }
    if (a.warm) {
        C<R>* out = (C<R>*)a.msg[a.ctl->cur];
        for (int t = threadIdx.x; t < D * CC; t += blockDim.x) {
            const int k = t / CC, r = t % CC;
            const int e = plain_slot_edge(sl, k);
            if (e < 0) continue;
            const int o = 2 * e + (a.edge_info[e].x == v ? 0 : 1);
            const int j = r / CHI, jp = r % CHI;
            out[(size_t)o * CC + r] = C<R>{(!MIX && j == jp) ? (R)m0[k][j] : (R)0, (R)0};
        }
    }
    if constexpr (MIX) {
        __shared__ cd F0[D][CC];
        __shared__ double tr0[D];
        __syncthreads();
        // PN lanes per entry (j <= j') of a slot
        constexpr int NU = CHI * (CHI + 1) / 2, PN = CHI == 16 ? 1 : (CHI == 4 ? 8 : 16), NO = H / CHI;
        for (int item = threadIdx.x / PN; item < D * NU; item += blockDim.x / PN) {
            const int k = item / NU, part = threadIdx.x % PN;
            int u = item % NU, j = 0;
            while (u >= CHI - j) { u -= CHI - j; ++j; }
            const int jp = j + u;
            cd f = cd{0.0, 0.0};
            if (plain_slot_edge(sl, k) >= 0 && m0[k][j] > 0.0 && m0[k][jp] > 0.0) {
                const int sk = ipow(CHI, D - 1 - k);
                for (int q = part; q < 2 * NO; q += PN) {
                    const int i = q / NO, c = q % NO;
                    const int base = i * H + (c / sk) * sk * CHI + c % sk;
                    const int tj = base + j * sk, tp = base + jp * sk;
                    f = cfmac(Tm[tp + tp / CC], Tm[tj + tj / CC], f);
                }
            }
            f.x = group_sum<PN>(f.x, group_mask<PN>());
            f.y = group_sum<PN>(f.y, group_mask<PN>());
            if (part == 0) {
                const double d = m0[k][j] * m0[k][jp];
                f = d > 0.0 ? (1.0 / sqrt(d)) * f : cd{0.0, 0.0};
                F0[k][j * CHI + jp] = f;
                F0[k][jp * CHI + j] = conj(f);
            }
        }
        __syncthreads();
        if (threadIdx.x < D) {
            double tr = 0.0;
            for (int j = 0; j < CHI; ++j) tr += F0[threadIdx.x][j * CHI + j].x;
            tr0[threadIdx.x] = tr;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < D * CC; t += blockDim.x) {
            const int k = t / CC, r = t % CC;
            const int e = plain_slot_edge(sl, k);
            if (e < 0) continue;
            const int o = 2 * e + (a.edge_info[e].x == v ? 0 : 1);
            const int j = r / CHI, jp = r % CHI;
            cd d = F0[k][r];
            if (j == jp) d.x -= m0[k][j] * tr0[k];
            ((C<R>*)a.D0)[(size_t)o * CC + r] = ccast<R>(d);
            if (r == 0) a.t0[o] = cd{tr0[k], 0.0};
        }
    }
}

// ---------------------------------------------------------------------------
// Flooding BP (App. B) of the plain path in one cooperative launch: sweeps of Eq.
// (local_consistency) until dist/|E| < tol or max_iter, decided on the device.
//
// Per sweep: (A) an item is one physical index i of one vertex.  With L_s = T x_0 m_0 .. x_{s-1}
// m_{s-1} and R_s = T x_{s+1} m_{s+1}^H .. x_{D-1} m_{D-1}^H the message out of slot s is
// F_s[j][j'] = sum L_s[.. j@s ..] conj(R_s[.. j'@s ..]), so that 2 (D - 1) contractions along one slot
// serve all D messages (instead of D (D - 1)).  A lane contracts (part of) a fiber: it
// reads the fiber's CHI elements once into registers and writes its outputs in place; the
// message's entries are shared-memory broadcasts.  Mixed mode (messages m = m0 + delta): the same
// with dL_{s+1} = dL_s x m_s + (T prod m0) x delta_s, likewise dR, and
// F_s - F_s(m0) = sum dL conj(R) + (L - dL) conj(dR).  The halves i = 0, 1 are added in (B), one
// warp per message: trace, normalisation (reading R10), new - old and its Frobenius norm, a lower
// bound of the trace norm; only a sweep whose sum of bounds falls under tol |E| (or the last one)
// is followed by (C), the exact trace norms.  Two grid barriers per sweep; the host is not
// involved.
//
// chi = 16 in FP64 is bound by the FP64 pipe (7 contraction-sized products of 2 CHI^4 per vertex);
// splitting a vertex by i lets three 64 KB buffers fit shared memory and balances 2n items over
// the SMs; indices beyond a bond's current dimension are skipped there.
// ---------------------------------------------------------------------------
struct PlainBPArgs {
    PlainArgs p;
    double tol;
    int max_iter;
    void* Fp;                 // [2][2m][CC] partial messages
    double* acc;              // [6]: bounds and exact distances, cycled over three sweeps
    unsigned long long* bar;
    int nblocks, bar_expect;
    long long spin_limit;
};

template <int CHI, int D, typename R, typename RC>
struct PlainTeam {   // shared memory of one team
    using S = PlainShape<CHI, D, R, RC>;
    C<R>* buf[4];
    C<R>* m;      // [D][CC] incoming messages
    C<R>* dm;     // mixed: incoming delta
    R* m0;        // [D][CHI]: mixed, warm-start diagonals
    int* dim;     // [D] dimensions of the bonds, [4 ..] outgoing message of each slot (-1)
    __device__ PlainTeam(unsigned char* base) {
        C<R>* p = reinterpret_cast<C<R>*>(base);
        for (int k = 0; k < 4; ++k) buf[k] = p + (k < S::NB ? k : 0) * S::PH;
        m = p + S::NB * S::PH;
        dm = m + (S::MIX ? D * S::CC : 0);
        m0 = reinterpret_cast<R*>(dm + D * S::CC);
        dim = reinterpret_cast<int*>(m0 + D * CHI);
    }
};

// product of the warm-start weights of the slots before (SUF: after) K at element index r
template <int CHI, int D, int K, bool SUF, typename R>
__device__ __forceinline__ R plain_weight(const R* m0, int r) {
    R w = (R)1;
#pragma unroll
    for (int k = 0; k < D; ++k)
        if (SUF ? k > K : k < K) w *= m0[k * CHI + (r / ipow(CHI, D - 1 - k)) % CHI];
    return w;
}

// dst = src contracted along slot K with m_K (SUF: m_K^H); mixed: + weight (T contracted with
// delta_K); FIRST: src is T (mixed: the first term is absent).  dst may be src.
template <int CHI, int D, typename R, typename RC, int K, bool SUF, bool FIRST>
__device__ __forceinline__ void plain_contract(const PlainTeam<CHI, D, R, RC>& tm, C<R>* dst, const C<R>* src, int tid,
                                               int team) {
    using S = PlainShape<CHI, D, R, RC>;
    constexpr int ST = ipow(CHI, D - 1 - K), NP = CHI / S::XO, CC = S::CC;
    const int fib = tid / NP, part = tid % NP;
    const int base = (fib / ST) * ST * CHI + fib % ST;
    const C<R>* T = tm.buf[0];
    bool on = tid < S::ITEMS;
    int rk = CHI;
    if constexpr (S::RANK) {   // degree 3: the two other indices of the fiber
        constexpr int o0 = K == 0 ? 1 : 0, o1 = K == 2 ? 1 : 2;
        rk = tm.dim[K];
        on = on && (base / ipow(CHI, D - 1 - o0)) % CHI < tm.dim[o0] && (base / ipow(CHI, D - 1 - o1)) % CHI < tm.dim[o1];
    }
    C<R> in[CHI], tin[S::MIX ? CHI : 1];
    if (on) {
#pragma unroll
        for (int q = 0; q < CHI; ++q) {
            const int r = base + q * ST;
            if (!(S::MIX && FIRST)) in[q] = src[r + r / CC];
            if constexpr (S::MIX) tin[q] = T[r + r / CC];
        }
    }
    team_bar<S::NT>(team);
    if (on) {
        const C<R>* m = tm.m + K * CC;
        const C<R>* dl = tm.dm + K * CC;
        R w = (R)1;
        if constexpr (S::MIX && !FIRST) w = plain_weight<CHI, D, K, SUF>(tm.m0, base);
        for (int xo = 0; xo < S::XO; ++xo) {
            const int x = part * S::XO + xo;
            if (S::RANK && x >= rk) break;
            C<R> acc = C<R>{(R)0, (R)0};
            if constexpr (S::MIX) {
#pragma unroll
                for (int q = 0; q < CHI; ++q) {
                    if (S::RANK && q >= rk) break;
                    acc = SUF ? cfmac(dl[x * CHI + q], tin[q], acc) : cfma(tin[q], dl[q * CHI + x], acc);
                }
                if constexpr (!FIRST) acc = w * acc;
            }
            if constexpr (!(S::MIX && FIRST)) {
#pragma unroll
                for (int q = 0; q < CHI; ++q) {
                    if (S::RANK && q >= rk) break;
                    acc = SUF ? cfmac(m[x * CHI + q], in[q], acc) : cfma(in[q], m[q * CHI + x], acc);
                }
            }
            const int r = base + x * ST;
            dst[r + r / CC] = acc;
        }
    }
    team_bar<S::NT>(team);
}

// Partial message out of slot K into Fp: L (and R) may be absent at the ends (LAST: R_K = T, dR = 0;
// K = 0: L_0 = T, dL = 0).
template <int CHI, int D, typename R, typename RC, int K>
__device__ __forceinline__ void plain_overlap(const PlainTeam<CHI, D, R, RC>& tm, const C<R>* L, const C<R>* Rt, int tid,
                                              C<R>* Fp) {
    using S = PlainShape<CHI, D, R, RC>;
    constexpr int ST = ipow(CHI, D - 1 - K), CC = S::CC, NO = S::H / CHI, PARTS = S::PARTS;
    const int out = tm.dim[4 + K];
    if (out < 0) return;   // the same for the team
    const int pr = tid / PARTS, part = tid % PARTS, j = pr / CHI, jp = pr % CHI;
    const C<R>* T = tm.buf[0];
    C<R> f = C<R>{(R)0, (R)0};
    auto term = [&](int base) {
        const int rj = base + j * ST, rp = base + jp * ST;
        const int pj = rj + rj / CC, pp = rp + rp / CC;
        if constexpr (!S::MIX) {
            f = cfmac(K == D - 1 ? T[pp] : Rt[pp], K == 0 ? T[pj] : L[pj], f);
        } else {
            if constexpr (K > 0) {
                C<R> y = T[pp];
                if constexpr (K < D - 1) y = plain_weight<CHI, D, K, true>(tm.m0, base) * y;
                f = cfmac(y, L[pj], f);
            }
            if constexpr (K < D - 1) {
                C<R> x = T[pj];
                if constexpr (K > 0) x = L[pj] + plain_weight<CHI, D, K, false>(tm.m0, base) * x;
                f = cfmac(Rt[pp], x, f);
            }
        }
    };
    if constexpr (S::RANK) {
        constexpr int o0 = K == 0 ? 1 : 0, o1 = K == 2 ? 1 : 2;
        constexpr int s0 = ipow(CHI, D - 1 - o0), s1 = ipow(CHI, D - 1 - o1);
        const int n0 = tm.dim[o0], n1 = tm.dim[o1], rk = tm.dim[K];
        if (j < rk && jp < rk)
            for (int u = part; u < n0; u += PARTS)
                for (int v = 0; v < n1; ++v) term(u * s0 + v * s1);
    } else {
        for (int c = part; c < NO; c += PARTS) term((c / ST) * ST * CHI + c % ST);
    }
    f.x = group_sum<PARTS>(f.x, group_mask<PARTS>());
    f.y = group_sum<PARTS>(f.y, group_mask<PARTS>());
    if (part == 0) Fp[(size_t)out * CC + pr] = f;
}

// (A): the three or four partial messages of item (v, i)
template <int CHI, int D, typename R, typename RC>
__device__ void plain_bp_item(const PlainBPArgs& a, int item, int cur, int tid, int team,
                              const PlainTeam<CHI, D, R, RC>& tm) {
    using S = PlainShape<CHI, D, R, RC>;
    constexpr int CC = S::CC, NT = S::NT;
    const int v = item >> 1, i = item & 1;
    const int4 sl = a.p.vslots[v];
    const C<R>* src = (const C<R>*)a.p.msg[cur];
    team_bar<NT>(team);   // the team may still read the previous item's buffers
    if (tid < D) {
        const int e = plain_slot_edge(sl, tid);
        int dim = 1;
        if (e >= 0) {
            dim = 0;
            // (a NaN counts: its index must reach the distance, which reports it)
            for (int q = 0; q < CHI; ++q) dim = __ldcg(a.p.lam + (size_t)e * CHI + q) <= 0.0 ? dim : q + 1;
        }
        tm.dim[tid] = dim;
        tm.dim[4 + tid] = e < 0 ? -1 : 2 * e + (a.p.edge_info[e].x == v ? 0 : 1);
    }
    const C<R>* Tg = (const C<R>*)a.p.T + (size_t)item * S::H;
    for (int t = tid; t < S::H; t += NT) tm.buf[0][t + t / CC] = Tg[t];
    for (int t = tid; t < D * CC; t += NT) {
        const int k = t / CC, r = t % CC, e = plain_slot_edge(sl, k), j = r / CHI, jp = r % CHI;
        C<R> mv = e >= 0 ? ldcg(src + (size_t)(2 * e + (a.p.edge_info[e].x == v ? 1 : 0)) * CC + r)
                         : C<R>{(R)(!S::MIX && r == 0 ? 1 : 0), (R)0};
        if constexpr (S::MIX) {
            tm.dm[t] = mv;
            if (j == jp) {
                RC s = 0.0;
                for (int q = 0; q < CHI; ++q) s += lam_get(a.p.lam, CHI, e, q);
                const R z = s > 0.0 ? (R)(lam_get(a.p.lam, CHI, e, j) * nr_rcp(s)) : (R)0;
                tm.m0[k * CHI + j] = z;
                mv.x += z;
            }
        }
        tm.m[t] = mv;
    }
    team_bar<NT>(team);
    C<R>* T = tm.buf[0];
    C<R>* A = tm.buf[1];
    C<R>* B = tm.buf[2];
    C<R>* Fp = (C<R>*)a.Fp + (size_t)i * 2 * a.p.m * CC;
    if constexpr (D == 3) {
        plain_contract<CHI, D, R, RC, 0, false, true>(tm, A, T, tid, team);    // L_1
        plain_contract<CHI, D, R, RC, 2, true, true>(tm, B, T, tid, team);     // R_1
        plain_overlap<CHI, D, R, RC, 1>(tm, A, B, tid, Fp);
        team_bar<NT>(team);
        plain_contract<CHI, D, R, RC, 1, false, false>(tm, A, A, tid, team);   // L_2
        plain_contract<CHI, D, R, RC, 1, true, false>(tm, B, B, tid, team);    // R_0
        plain_overlap<CHI, D, R, RC, 2>(tm, A, T, tid, Fp);
        plain_overlap<CHI, D, R, RC, 0>(tm, T, B, tid, Fp);
    } else {
        C<R>* E = tm.buf[3];
        plain_contract<CHI, D, R, RC, 0, false, true>(tm, A, T, tid, team);    // L_1
        plain_contract<CHI, D, R, RC, 3, true, true>(tm, B, T, tid, team);     // R_2
        plain_contract<CHI, D, R, RC, 2, true, false>(tm, E, B, tid, team);    // R_1
        plain_overlap<CHI, D, R, RC, 1>(tm, A, E, tid, Fp);
        team_bar<NT>(team);
        plain_contract<CHI, D, R, RC, 1, false, false>(tm, A, A, tid, team);   // L_2
        plain_contract<CHI, D, R, RC, 1, true, false>(tm, E, E, tid, team);    // R_0
        plain_overlap<CHI, D, R, RC, 2>(tm, A, B, tid, Fp);
        plain_overlap<CHI, D, R, RC, 0>(tm, T, E, tid, Fp);
        team_bar<NT>(team);
        plain_contract<CHI, D, R, RC, 2, false, false>(tm, A, A, tid, team);   // L_3
        plain_overlap<CHI, D, R, RC, 3>(tm, A, T, tid, Fp);
    }
}

// sqrt of a squared norm, 0 for 0; a NaN stays one, so that the distance reports it
template <typename R>
__device__ __forceinline__ R norm_root(R x) {
    return x == x ? nr_sqrt(x) : x;
}

// (B): message o from its two halves; returns the Frobenius norm of new - old
template <int CHI, typename R, typename RC>
__device__ RC plain_bp_finish(const PlainBPArgs& a, int o, int cur, int lane) {
    constexpr int CC = CHI * CHI, NE = (CC + 31) / 32;
    constexpr bool MIX = sizeof(R) != sizeof(RC);
    const C<R>* F0 = (const C<R>*)a.Fp + (size_t)o * CC;
    const C<R>* F1 = F0 + (size_t)2 * a.p.m * CC;
    const C<R>* old = (const C<R>*)a.p.msg[cur] + (size_t)o * CC;
    C<R>* dst = (C<R>*)a.p.msg[cur ^ 1] + (size_t)o * CC;
    C<RC> f[NE];
    RC tr[3] = {(RC)0, (RC)0, (RC)0};   // trace, and sum(lambda)
#pragma unroll
    for (int q = 0; q < NE; ++q) {
        const int r = lane + 32 * q;
        f[q] = C<RC>{(RC)0, (RC)0};
        if (r < CC) {
            f[q] = ccast<RC>(ldcg(F0 + r)) + ccast<RC>(ldcg(F1 + r));
            if (r / CHI == r % CHI) {
                tr[0] += f[q].x;
                tr[1] += f[q].y;
            }
        }
    }
    RC lam = (RC)0;
    if constexpr (MIX) {
        if (lane < CHI) lam = __ldcg(a.p.lam + (size_t)(o >> 1) * CHI + lane);
        tr[2] = lam;
    }
    group_sums<32>(tr, 0xffffffffu);
    C<RC> den = C<RC>{tr[0], tr[1]};
    if constexpr (MIX) den = den + ldcg(a.p.t0 + o);
    const RC n2 = norm2(den);
    const RC in = n2 > (RC)0 ? nr_rcp(n2) : (RC)0;
    const C<RC> itr = C<RC>{den.x * in, -den.y * in};
    const RC m0 = MIX && tr[2] > (RC)0 ? lam * nr_rcp(tr[2]) : (RC)0;   // lane j: m0_j
    RC d2 = (RC)0;
#pragma unroll
    for (int q = 0; q < NE; ++q) {
        const int r = lane + 32 * q, j = r / CHI, jp = r % CHI;
        C<RC> num = f[q];
        if constexpr (MIX) {
            const RC z = __shfl_sync(0xffffffffu, m0, j & 31);
            if (r < CC) {
                num = num + ccast<RC>(ldcg((const C<R>*)a.p.D0 + (size_t)o * CC + r));
                if (j == jp) num = num - z * C<RC>{tr[0], tr[1]};
            }
        }
        if (r < CC) {
            const C<RC> nv = num * itr;
            const C<RC> d = nv - ccast<RC>(ldcg(old + r));
            dst[r] = ccast<R>(nv);
            ((C<R>*)a.p.dm)[(size_t)o * CC + r] = ccast<R>(d);
            d2 += norm2(d);
        }
    }
    d2 = group_sum<32>(d2, 0xffffffffu);
    return norm_root(d2);
}

// (C): trace norm of new - old of message o (group of CC / 2 lanes)
template <int CHI, typename R, typename RC, typename Group>
__device__ RC plain_trace_norm(const C<R>* dm, unsigned char* base, int g, const Group& grp) {
    constexpr int CC = CHI * CHI, GL = CC / 2;
    C<RC>* A = reinterpret_cast<C<RC>*>(base);
    for (int t = g; t < CC; t += GL) A[t] = ccast<RC>(ldcg(dm + t));
    grp.sync();
    RC s = (RC)0;
    if constexpr (sizeof(RC) == 8) {
        cd* V = A + CC;
        cd* T = V + CC;
        cf* A32 = reinterpret_cast<cf*>(T + CC);
        double* nrm = reinterpret_cast<double*>(A32 + 2 * CC);
        prune_noise<CHI>(A, g, grp);
        // tol 1e-8: the sum of the values depends on a cosine that is left only in second order, so pairs
        // of close lengths (a traceless difference has them) need no rotation beyond that
        refined_svd<CHI, true>(A, V, A32, A32 + CC, T, nrm, nullptr, g, grp, group_mask<CHI>(), 1e-16, CHI, 1e-8f, 1e-8);
        if (g == 0)
            for (int q = 0; q < CHI; ++q) s += norm_root(nrm[q]);
    } else {
        jacobi_svd<CHI, RC, Group, false>(A, nullptr, g, grp, group_mask<CHI>(), (RC)1e-6, 60, false);
        grp.sync();
        if (g == 0)
            for (int q = 0; q < CHI; ++q) {
                RC n2 = (RC)0;
                for (int r = 0; r < CHI; ++r) n2 += norm2(A[q * CHI + r]);
                s += norm_root(n2);
            }
    }
    grp.sync();
    return s;
}

template <int CHI, int D, typename R, typename RC>
__global__ void __launch_bounds__(512, 1) plain_bp_kernel(PlainBPArgs a) {
    using S = PlainShape<CHI, D, R, RC>;
    constexpr int CC = S::CC, NT = S::NT, GL = S::GL;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    __shared__ double bsum;
    __shared__ int flags[8];
    Control* ctl = a.p.ctl;
    if (threadIdx.x == 0) flags[0] = run_failed(ctl);   // one value per block: another one may give up meanwhile
    GridBarrier gb = grid_barrier_init(a.bar, &ctl->err, (unsigned)a.bar_expect);
    int cur = *(volatile int*)&ctl->cur;
    const int team = threadIdx.x / NT, tid = threadIdx.x % NT;
    const PlainTeam<CHI, D, R, RC> tm(plain_smem + team * ((S::team_smem + 15) / 16 * 16));
    const double E = (double)a.p.m, slack = sizeof(R) == 4 ? 1e-5 : 1e-12;
    const double go = a.tol * E / (1.0 - slack);   // a bound at least this large cannot stop
    double dist = 0.0;
    bool conv = false;
    int it = 0;
    // the accumulators of sweep `it` are zeroed two barriers ahead (those of the first sweeps by the host)
    while (it < a.max_iter) {
        double* acc = a.acc + it % 3;
        double* ex = a.acc + 3 + it % 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.acc[(it + 1) % 3] = 0.0;
            a.acc[3 + (it + 1) % 3] = 0.0;
        }
        for (int item = team * a.nblocks + blockIdx.x; item < 2 * a.p.n; item += a.nblocks * S::TEAMS)
            plain_bp_item<CHI, D, R, RC>(a, item, cur, tid, team, tm);
        if (it == 0) {
            __syncthreads();
            if (flags[0]) return;
        }
        if (!grid_sync(gb, a.spin_limit)) return;
        if (threadIdx.x == 0) bsum = 0.0;
        __syncthreads();
        double mine = 0.0;
        for (int o = (threadIdx.x / 32) * a.nblocks + blockIdx.x; o < 2 * a.p.m; o += a.nblocks * (S::TPB / 32))
            mine += (double)plain_bp_finish<CHI, R, RC>(a, o, cur, threadIdx.x & 31);
        if ((threadIdx.x & 31) == 0 && mine != 0.0) atomicAdd(&bsum, mine);
        __syncthreads();
        if (threadIdx.x == 0 && bsum != 0.0) atomicAdd(acc, bsum);
        if (!grid_sync(gb, a.spin_limit)) return;
        cur ^= 1;
        ++it;
        const bool last = it >= a.max_iter;
        const double bound = __ldcg(acc);
        if (!(bound == bound)) {
            dist = bound;
            break;
        }
        if (!last && a.p.m > 0 && bound >= go) continue;
        if (threadIdx.x == 0) bsum = 0.0;
        __syncthreads();
        const int gi = threadIdx.x / GL, g = threadIdx.x % GL;
        if (gi < S::GROUPS) {
            unsigned char* base = plain_smem + gi * ((S::group_smem + 15) / 16 * 16);
            double t = 0.0;
            for (int o = gi * a.nblocks + blockIdx.x; o < 2 * a.p.m; o += a.nblocks * S::GROUPS) {
                const C<R>* dm = (const C<R>*)a.p.dm + (size_t)o * CC;
                if constexpr (GL <= 32) t += (double)plain_trace_norm<CHI, R, RC>(dm, base, g, WarpGroup{group_mask<GL>()});
                else t += (double)plain_trace_norm<CHI, R, RC>(dm, base, g, TeamGroup<GL>{gi, &flags[gi]});
            }
            if (g == 0 && t != 0.0) atomicAdd(&bsum, t);
        }
        __syncthreads();
        if (threadIdx.x == 0 && bsum != 0.0) atomicAdd(ex, bsum);
        if (blockIdx.x == 0 && threadIdx.x == 0) ++ctl->exact_passes;
        if (!grid_sync(gb, a.spin_limit)) return;
        dist = a.p.m > 0 ? __ldcg(ex) / E : 0.0;
        if (!(dist == dist)) break;
        if (dist < a.tol) {
            conv = true;
            break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (!(dist == dist)) ctl->err = 3;   // GTQA_ERR_NUMERIC
        ctl->last_iters = it;
        ctl->last_dist = dist;
        ctl->not_conv = conv ? 0 : 1;
        ctl->sweeps_total += it;
        ctl->bp_calls += 1;
        ctl->nc_calls += conv ? 0 : 1;
        ctl->cur = cur;
    }
}

// Vidal gauge finding, edge part (App. D "Vidal gauge finding"), block = CHI^2 threads:
// Hermitian eigen-decompositions of m_{a->b} and m_{b->a} (as SVDs, each by half of the block; signs
// from v^H A v), principal square roots and pseudo-inverse square roots, the SVD of
// M = (m_{a->b}^{1/2})^T m_{b->a}^{1/2}, lambda = S/||S||, X_a = conj(m_{a->b}^{-1/2}) U ||S||^{1/2}
// and X_b = conj(m_{b->a}^{-1/2}) V^* ||S||^{1/2}.
template <int CHI, typename RC>
struct PlainEdgeSm {
    static constexpr int CC = CHI * CHI;
    C<RC> Am[2][CC], Vm[2][CC], Y[2][CC], M[CC], VM[CC];
    C<RC> T[2][sizeof(RC) == 8 ? CC : 1];
    cf A32[2][sizeof(RC) == 8 ? CC : 1], V32[2][sizeof(RC) == 8 ? CC : 1];
    double n2[2][CHI];
    RC w[2][CHI], wq[2][CHI], wiq[2][CHI], sig[CHI], isig[CHI], m0[CHI], scal[2];
    int perm[CHI], flag[2];
};
template <int CHI, typename RC, typename Group>
__device__ __forceinline__ void plain_edge_svd(C<RC>* A, C<RC>* V, PlainEdgeSm<CHI, RC>& sm, int x, int g,
                                               const Group& grp, double cut) {
    if constexpr (sizeof(RC) == 8) {
        prune_noise<CHI>(A, g, grp);
        refined_svd<CHI, true>(A, V, sm.A32[x], sm.V32[x], sm.T[x], sm.n2[x], nullptr, g, grp, group_mask<CHI>(), cut, CHI,
                               1e-8f, 1e-15);
    } else if constexpr (CHI * CHI / 2 <= 32) {
        jacobi_v32<CHI, true>(A, V, g, group_mask<CHI * CHI / 2>(), group_mask<CHI>(), CHI);
        grp.sync();
    } else {
        jacobi_svd<CHI, RC>(A, V, g, grp, group_mask<CHI>(), (RC)1e-6, 60, true, nullptr, (RC)1e-3);
    }
}
template <int CHI, typename R, typename RC = R>
__global__ void __launch_bounds__(CHI * CHI) plain_regauge_edge_kernel(PlainArgs a, double eig_cut, double svd_cut) {
    constexpr int CC = CHI * CHI, GL = CC / 2, NT = CC;
    constexpr bool MIX = sizeof(R) != sizeof(RC);
    extern __shared__ __align__(16) unsigned char plain_smem[];
    PlainEdgeSm<CHI, RC>& sm = *reinterpret_cast<PlainEdgeSm<CHI, RC>*>(plain_smem);
    const int e = blockIdx.x, tid = threadIdx.x;
    auto bar = [&]() {
        if constexpr (NT < 32) __syncwarp(group_mask<NT>());
        else __syncthreads();
    };
    auto half_svd = [&](C<RC>* A, C<RC>* V, int x, int g, double cut) {
        if constexpr (GL <= 32) plain_edge_svd<CHI, RC>(A, V, sm, x, g, WarpGroup{group_mask<GL>()}, cut);
        else plain_edge_svd<CHI, RC>(A, V, sm, x, g, TeamGroup<GL>{x, &sm.flag[x]}, cut);
    };
    const bool failed = run_failed(a.ctl);
    const C<R>* msg = (const C<R>*)a.msg[a.ctl->cur];
    // mixed mode: the messages hold delta = m - m0, m0 = diag(lambda_e)/sum(lambda_e) (read before
    // this kernel overwrites lambda_e)
    if (MIX && tid < CHI) {
        RC sum = 0.0;
        for (int q = 0; q < CHI; ++q) sum += a.lam[(size_t)e * CHI + q];
        sm.m0[tid] = sum > 0.0 ? a.lam[(size_t)e * CHI + tid] / sum : 0.0;
    }
    if (MIX) bar();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC;
        const int row = r % CHI, col = r / CHI;
        const C<R>* mm = msg + (size_t)(2 * e + x) * CC;
        C<RC> v = ccast<RC>(mm[row * CHI + col]), vt = ccast<RC>(mm[col * CHI + row]);
        if (MIX && row == col) {
            v.x += sm.m0[row];
            vt.x += sm.m0[row];
        }
        sm.Am[x][col * CHI + row] = C<RC>{(RC)0.5 * (v.x + vt.x), (RC)0.5 * (v.y - vt.y)};
    }
    bar();
    half_svd(sm.Am[tid / GL], sm.Vm[tid / GL], tid / GL, tid % GL, eig_cut);
    bar();
    for (int t = tid; t < 2 * CHI; t += NT) {
        const int x = t / CHI, k = t % CHI;
        RC n2 = 0.0, sg = 0.0;
        for (int r = 0; r < CHI; ++r) {
            const C<RC> av = sm.Am[x][k * CHI + r], vv = sm.Vm[x][k * CHI + r];
            n2 += norm2(av);
            sg += vv.x * av.x + vv.y * av.y;
        }
        const RC wv = nr_sqrt(n2);
        sm.w[x][k] = sg >= 0.0 ? wv : -wv;
    }
    bar();
    for (int t = tid; t < 2 * CHI; t += NT) {   // the roots of each kept eigenvalue once
        const int x = t / CHI, k = t % CHI;
        RC wmax = 0.0;
        for (int q = 0; q < CHI; ++q) wmax = fmax(wmax, sm.w[x][q]);
        const RC wk = sm.w[x][k];
        const RC is = wk > eig_cut * wmax ? nr_rsqrt(wk) : (RC)0;
        sm.wiq[x][k] = is;
        sm.wq[x][k] = is > (RC)0 ? wk * is : (RC)0;
    }
    bar();
    // with m_x = V_x w_x V_x^H: M = conj(V_0) B V_1^H, B = w_0^{1/2} (V_0^T V_1) w_1^{1/2}; with the SVD of
    // B the transforms are conj(V_x) w_x^{-1/2} times its scaled singular vectors (as on the persistent path)
    for (int t = tid; t < CC; t += NT) {
        const int k = t % CHI, l = t / CHI;
        C<RC> acc = C<RC>{(RC)0, (RC)0};
        for (int j = 0; j < CHI; ++j) acc = cfma(sm.Vm[0][k * CHI + j], sm.Vm[1][l * CHI + j], acc);
        sm.M[l * CHI + k] = (sm.wq[0][k] * sm.wq[1][l]) * acc;
    }
    bar();
    if (tid < GL) half_svd(sm.M, sm.VM, 0, tid, svd_cut);
    bar();
    for (int cc = tid; cc < CHI; cc += NT) {
        RC n2 = 0.0;
        for (int r = 0; r < CHI; ++r) n2 += norm2(sm.M[cc * CHI + r]);
        const RC sv = nr_sqrt(n2);
        sm.sig[cc] = sv;
        sm.isig[cc] = sv > (RC)0 ? nr_rcp(sv) : (RC)0;
    }
    bar();
    for (int cc = tid; cc < CHI; cc += NT) sm.perm[desc_rank(sm.sig, CHI, cc)] = cc;
    if (failed) return;
    bar();
    if (tid == 0) {
        RC tot = 0.0;
        for (int cc = 0; cc < CHI; ++cc) tot += sm.sig[cc] * sm.sig[cc];
        const RC nrm = nr_sqrt(tot);
        sm.scal[0] = nrm;
        sm.scal[1] = nr_sqrt(nrm);
        const RC inrm = nrm > 0.0 ? nr_rcp(nrm) : 0.0;
        const RC smax = sm.sig[sm.perm[0]];
        for (int r = 0; r < CHI; ++r) {
            const RC s = sm.sig[sm.perm[r]];
            a.lam[(size_t)e * CHI + r] = (nrm > 0.0 && s > svd_cut * smax) ? s * inrm : 0.0;
        }
    }
    bar();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC, j = r / CHI, k = r % CHI;
        const int pc = sm.perm[j];
        const bool kept = sm.scal[0] > 0.0 && sm.sig[pc] > svd_cut * sm.sig[sm.perm[0]];
        const RC f = kept ? sm.wiq[x][k] * sm.scal[1] : (RC)0;
        sm.Y[x][r] = x == 0 ? (f * sm.isig[pc]) * sm.M[pc * CHI + k] : f * conj(sm.VM[pc * CHI + k]);
    }
    bar();
    for (int t = tid; t < 2 * CC; t += NT) {
        const int x = t / CC, r = t % CC, jpp = r / CHI, j = r % CHI;
        C<RC> acc = C<RC>{(RC)0, (RC)0};
        for (int k = 0; k < CHI; ++k) acc = cfmac(sm.Vm[x][k * CHI + jpp], sm.Y[x][j * CHI + k], acc);
        ((C<R>*)a.X)[((size_t)e * 2 + x) * CC + r] = ccast<R>(acc);
    }
}

// Vidal gauge finding, vertex part: Gamma[.., j@k, ..] = sum_q T[.., q@k, ..] X_k[q][j] for every
// slot (X of the edge, from this vertex's side; identity on phantom slots).  One block per (vertex,
// physical index); a lane contracts (part of) a fiber in place.
template <int CHI, int D, typename R, int K>
__device__ __forceinline__ void plain_regauge_slot(C<R>* buf, C<R>* Xs, const PlainArgs& a, const int4& sl, int v, int tid) {
    if constexpr (K < D) {
        using S = PlainShape<CHI, D, R, R>;
        constexpr int ST = ipow(CHI, D - 1 - K), NP = CHI / S::XO, CC = S::CC, NT = S::NT;
        const int e = plain_slot_edge(sl, K);
        if (e >= 0) {   // the same for the block
            const int side = a.edge_info[e].x == v ? 0 : 1;
            for (int t = tid; t < CC; t += NT) Xs[t] = ((const C<R>*)a.X)[((size_t)e * 2 + side) * CC + t];
            const int fib = tid / NP, part = tid % NP, base = (fib / ST) * ST * CHI + fib % ST;
            C<R> in[CHI];
            bool any = false;
            if (tid < S::ITEMS) {
#pragma unroll
                for (int q = 0; q < CHI; ++q) {
                    const int r = base + q * ST;
                    in[q] = buf[r + r / CC];
                    any |= in[q].x != (R)0 || in[q].y != (R)0;
                }
            }
            __syncthreads();
            if (any)   // a fiber of zeros stays one (indices beyond the bonds' dimensions)
                for (int xo = 0; xo < S::XO; ++xo) {
                    const int x = part * S::XO + xo;
                    C<R> acc = C<R>{(R)0, (R)0};
#pragma unroll
                    for (int q = 0; q < CHI; ++q) acc = cfma(in[q], Xs[q * CHI + x], acc);
                    const int r = base + x * ST;
                    buf[r + r / CC] = acc;
                }
            __syncthreads();
        }
        plain_regauge_slot<CHI, D, R, K + 1>(buf, Xs, a, sl, v, tid);
    }
}
template <int CHI, int D, typename R>
__global__ void __launch_bounds__(PlainShape<CHI, D, R, R>::NT) plain_regauge_vertex_kernel(PlainArgs a) {
    using S = PlainShape<CHI, D, R, R>;
    constexpr int CC = S::CC, NT = S::NT;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    C<R>* buf = reinterpret_cast<C<R>*>(plain_smem);
    C<R>* Xs = buf + S::PH;
    const int v = blockIdx.x >> 1;
    const int4 sl = a.vslots[v];
    const bool failed = run_failed(a.ctl);
    const C<R>* T = (const C<R>*)a.T + (size_t)blockIdx.x * S::H;
    for (int t = threadIdx.x; t < S::H; t += NT) buf[t + t / CC] = T[t];
    __syncthreads();
    plain_regauge_slot<CHI, D, R, 0>(buf, Xs, a, sl, v, threadIdx.x);
    if (failed) return;
    C<R>* g = (C<R>*)a.Gamma + (size_t)blockIdx.x * S::H;
    for (int t = threadIdx.x; t < S::H; t += NT) g[t] = buf[t + t / CC];
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
    C<R> T[sizeof(R) == 8 ? S::NM * S::NM : (S::LS > 32 ? 2 * S::NM * S::NM : 1)];   // scratch of the SVD
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
    static_assert(G >= CHI, "lane l holds row l of R");
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
    CR T[(sizeof(R) == 8 ? 1 : 2) * NM * NM];   // scratch of the SVD; then Z [block][j][col]
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
    for (int j = 0; j < CHI; ++j) nc = sm.lab[j] <= 0.0 ? nc : j + 1;   // (a NaN counts)
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
