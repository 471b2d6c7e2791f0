// Persistent annealing kernel: one cooperative launch runs whole GTQA layers.
//
// Phases of one layer (each separated by a bounded grid barrier):
//   gates      for each colour class: simple update + truncation of every edge of
//              that matching (App. E, App. D "Truncation"); the mixing gate
//              exp(-i t_X X) (Sec. II D) is applied to a vertex right after its last
//              gate of the layer, and a leading mixing gate exp(-i t_pre X) (the
//              second-order and reversed first-order product formulas of Sec. V)
//              right before its first gate.
//   bp init    T_a = Gamma_a prod lambda^{1/2} (Eq. (symmetric_gauge)); warm-start
//              messages diag(lambda)/sum(lambda) (Eq. (reconstructed_messages)).
//   bp sweeps  flooding update of every directed message, Eq. (local_consistency),
//              unit-trace normalisation and trace-norm distance (App. B), until
//              dist_b/|E_b| < tol for every instance b or max_iter sweeps.
//   regauge    Vidal gauge finding (App. D): per-edge transforms, then per-vertex
//              application to T.
//
// Layout: Gamma[n][2][CHI][CHI][CHI] (slot k = k-th incident edge, ascending id),
// lambda[m][CHI], messages[2m][CHI][CHI] (2e = m_{u->v}, 2e+1 = m_{v->u}); phantom
// slots (degree < 3) have dimension 1 with lambda = e_0 and message e_0 e_0^T.
//
// Precision modes:
//   FP64   complex128 tensors and messages, FP64 arithmetic throughout.
//   Mixed  complex64 Gamma, T and message corrections; the simple update's QR and
//          SVD and the regauge's eigen/SVD and square roots in FP64 (first stage and
//          small corrections of the SVDs in FP32), the message normalisation from
//          pairs of floats (1e-13).  Messages are kept as m = m0 + delta with m0 the
//          warm start (exact, from lambda) and delta in complex64; each sweep
//          contracts only delta in FP32, and the warm-start part F(m0) is contracted
//          once per BP call in FP64.
#pragma once

#include <type_traits>

#include "gtqa_common.cuh"

namespace gtqa {

struct ModeFP64 {
    using TS = double;   // storage of Gamma, T, messages
    using RC = double;   // arithmetic of the SVDs, QRs and gauge roots
    static constexpr bool mixed = false;
};
struct ModeMixed {
    using TS = float;
    using RC = double;
    static constexpr bool mixed = true;
};
// every step in complex64 / FP32 (a reference point for the precision split; plain kernels only)
struct ModeC64 {
    using TS = float;
    using RC = float;
    static constexpr bool mixed = false;
};

enum : unsigned { PH_GATES = 1u, PH_BP = 2u, PH_WARM = 4u, PH_REGAUGE = 8u };

struct Control {
    unsigned long long bar_count;   // grid-barrier arrivals (monotonic), a multiple of the grid between launches
    unsigned long long bar_pk[3];   // the same, one counter per phase kernel (each kernel keeps its grid size)
    int err;
    int cur;                 // message buffer holding the latest messages
    long long sweeps_total;  // sum over BP calls of max-over-instances sweeps
    int last_iters;          // sweeps of the last BP call (max over instances)
    int not_conv;            // instances at max_iter in the last BP call
    double last_dist;        // max over instances of the final dist/|E|
    long long bp_calls;
    long long nc_calls;      // BP calls in which some instance hit max_iter
    long long regauged;      // regauge-policy layers: regauged (BP and gauge finding ran)
    long long reg_skipped;   // and skipped (R at or below the threshold)
    long long exact_passes;  // separate exact-distance passes (bp_exact_pass) run by BP
    int gate_sw_max;         // most FP64 refinement passes of one gate-core SVD (and sweeps of its closing polish)
    int gate_sw32_max;       // most FP32 Jacobi sweeps of one gate-core SVD
    int reg_sw_max;          // the same for the regauge's eigen-decompositions and SVD
    int reg_sw32_max;
};

struct Ctx {
    // graph
    const int4* edge_info;    // u, v, slot in u, slot in v
    const int4* vert_edges;   // edge at slots 0..2 (-1 phantom), degree
    const int* vert_inst;
    const double* J;
    const double* hd;         // h_a / degree of a
    const struct GateMeta* gates;   // [m], colour by colour
    const int* colour_off;    // [ncol + 1]
    const int* iso;           // vertices of degree 0
    int n_iso;
    int ncol;
    int n, m, B;
    const int* inst_vbeg;     // [B + 1]
    const int* inst_m;
    // state
    void* Gamma;
    double* lam;
    void* T;
    void* msg[2];
    cf* D0;                   // mixed: warm-start defect F(m0) - tr F(m0) m0, [2m][CHI^2]
    float4* t0;               // mixed: tr F(m0) as a sum of two complex floats, [2m]
    float* m0f;               // mixed: the warm-start diagonal of each message, [2m][CHI]
    cd* X;                    // regauge transforms [m][2][CHI^2]
    double* acc;              // [3][B] per-sweep distance accumulators
    int* inst_done;
    int* inst_iters;
    double* inst_dist;
    double* stats;            // discarded weight, log fidelity, gate SVD pairs and rotations, regauge SVD sweeps
    Control* ctl;
    unsigned long long* bar;  // barrier counter of this launch (null: ctl->bar_count)
    // parameters
    int chi;
    double svd_cut, eig_cut;
    double tol;
    int max_iter;
    unsigned phases;
    int k0, k1, Ksched;       // layers k0..k1 with tau = k/Ksched; Ksched = 0: one layer at (tZ1, tX1)
    int* kdev;                // non-null: one layer, k read from *kdev; the regauge phase stores k + 1
                              // (CUDA-graph replays of one captured layer advance through the anneal)
    double dt, tZ1, tX1;
    double tXpre1;            // Ksched = 0: leading mixing angle of the layer (0: none)
    const double* rgate;      // regauge policy: the residual sum of this layer (null: always regauge)
    double rthr_sum;          // BP and regauge run only if *rgate > rthr_sum
    int nblocks;
    int nsm;                  // SMs of the device: the team widths follow it, not the grid, so that a grid
                              // chosen by gtqa_set_grid or gtqa_autotune does not change the rounding
    int bar_expect;           // arrivals per grid barrier (= nblocks; larger only in the timeout test)
    long long spin_limit;
};

template <int CHI> __host__ __device__ constexpr int sstride(int k) {
    return k == 0 ? CHI * CHI : (k == 1 ? CHI : 1);
}
__host__ __device__ inline void others_of(int s, int& o0, int& o1) {
    o0 = (s == 0) ? 1 : 0;
    o1 = (s == 2) ? 1 : 2;
}
__device__ __forceinline__ double lam_get(const double* lam, int CHI, int e, int j) {
    return e < 0 ? (j == 0 ? 1.0 : 0.0) : __ldcg(lam + (size_t)e * CHI + j);
}

// Launch shapes of the persistent phase kernels: threads per block and team sizes.  The gate
// team TG (one lane per element pair of the Jacobi SVD of the 2CHI x 2CHI core), the
// regauge-edge team TR and the BP-init team TV are fixed by their algorithms; the block size
// TPB, the BP vertex team TB and the regauge-vertex team TRV come in NSHAPE variants, which
// gtqa_autotune times kernel by kernel.  Variant 0 is the default, at CHI = 8 variant 1 on large instances:
//   CHI <= 4: (TPB, TB, TRV) = (512, 64, 32), (256, 64, 32), (512, 128, 64)
//   CHI  = 8:                  (256, 256, 128), (512, 256, 128), (512, 512, 256)
constexpr int NSHAPE = 3;
template <int CHI, int V = 0> struct Shape {
    static_assert(V >= 0 && V < NSHAPE, "launch-shape variant");
    static constexpr bool BIG = CHI >= 8;
    static constexpr int TPB = V == 0 ? (BIG ? 256 : 512) : (V == 1 ? (BIG ? 512 : 256) : 512);
    static constexpr int TG = 2 * CHI * CHI;                                           // gate team
    static constexpr int TB = V == 2 ? (BIG ? 512 : 128) : (BIG ? 256 : 64);            // BP team (one vertex)
    static constexpr int TR = CHI * CHI;                                               // regauge-edge team
    static constexpr int TV = 32;                                                      // BP-init team (one warp)
    // warps of a block that run the BP init (its per-warp scratch grows as CHI^3)
    static constexpr int NIT = BIG && TPB / 32 > 8 ? 8 : TPB / 32;
    static constexpr int TRV = V == 2 ? (BIG ? 256 : 64) : (BIG ? 128 : 32);           // regauge-vertex team
};

// ===========================================================================
// gates: simple update of one edge (team of 2 CHI^2 threads)
//
// The FP64 pipe bounds it (64 cycles per warp instruction and sub-partition): at n = 1000,
// chi = 4 every sub-partition holds one gate of a colour, so the time of a phase is the FP64
// instruction count of a gate plus the latencies in between.  Hence: the four QRs keep their rows
// in registers, all inner products of a reflector are summed at once (group_sums), scalars are
// formed once per group of lanes, and the reflectors go to shared memory already scaled, in the
// type of the back-application.
// ===========================================================================
// One gate of the schedule, in the order the colours run: everything a team has to know before it
// touches the state.
struct GateMeta {
    int4 a;   // edge, u, v, bits: slot in u, slot in v (two each); first gate of u, of v; last of u, of v
    int4 b;   // edges at the other slots of u and of v, ascending (-1: none)
};

template <int CHI, class Mode>
struct GateSm {
    using TS = typename Mode::TS;
    static constexpr int PB = CHI == 2 ? 2 : 8;   // four lanes each
    C<TS> U[4][CHI][CHI * CHI];   // [block][col][row]: scaled reflectors, then the new tensors
    cd M[4 * CHI * CHI];
    cd V[4 * CHI * CHI];       // first the R factors [block][row][col], then V
    cd G[4 * CHI * CHI];       // scratch of the refinement
    cf M32[4 * CHI * CHI];     // FP32 copy of M for the first stage
    cf V32[4 * CHI * CHI];
    double lab[CHI];
    double sig[2 * CHI];
    double isig[2 * CHI];      // 1 / sig
    cd phases[PB * 4];         // diagonal gate phases of the team's next PB gates
    int perm[2 * CHI];
    int keep;
    unsigned relmask;          // columns that decide the stop of a closing polish
    int flag;
    int nrot;
};

// Householder steps K .. CHI - 1 of a (2 G) x CHI block, rows l and l + G of a lane in y0, y1.
// The reflector of step k is stored as u = sqrt(tau) v (|u| = sqrt 2) in the type of the
// back-application, [col][row]; y0 of the lanes l < CHI ends as the rows of R.
template <int CHI, int G, int K, typename R, typename RB>
__device__ __forceinline__ void qr_steps(C<R> (&y0)[CHI], C<R> (&y1)[CHI], C<RB>* U, int l, unsigned gm) {
    if constexpr (K < CHI) {
        using CR = C<R>;
        constexpr int NC = CHI - 1 - K;   // later columns
        const CR z = CR{(R)0, (R)0};
        const CR x0 = l >= K ? y0[K] : z, x1 = y1[K];
        // |x|^2 and x^H y of every later column
        R s[1 + 2 * NC];
        s[0] = fma(x0.x, x0.x, fma(x0.y, x0.y, fma(x1.x, x1.x, x1.y * x1.y)));
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const CR d = cfmac(x0, y0[K + 1 + c], cfmac(x1, y1[K + 1 + c], z));
            s[1 + 2 * c] = d.x;
            s[2 + 2 * c] = d.y;
        }
        group_sums<G>(s, gm);
        const CR xkk = CR{__shfl_sync(gm, y0[K].x, K, G), __shfl_sync(gm, y0[K].y, K, G)};
        const R a2 = norm2(xkk);
        // 1 / |x| on the even lanes and 1 / |x_K| on the odd ones, in one pass of the pipe
        const R arg = (l & 1) ? a2 : s[0];
        const R rs = arg > tiny_norm2<R>() ? nr_rsqrt(arg) : (R)0;
        const R r0 = __shfl_sync(gm, rs, 0, G), ra = __shfl_sync(gm, rs, 1, G);
        const R nrm = s[0] * r0, axkk = a2 * ra;
        const CR ph = nonzero(ra) ? CR{xkk.x * ra, xkk.y * ra} : CR{(R)1, (R)0};
        const R stau = nonzero(nrm) ? nr_rsqrt(nrm * (nrm + axkk)) : (R)0;
        const CR pv = nrm * ph;
        const CR vkk = xkk + pv;
        // tau v^H y = tau (x^H y + conj(|x| ph) y_K), column K + 1 + c on lane c
        CR sx = z, yk = z;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const R yx = __shfl_sync(gm, y0[K + 1 + c].x, K, G), yy = __shfl_sync(gm, y0[K + 1 + c].y, K, G);
            if (l % CHI == c) {
                sx = CR{s[1 + 2 * c], s[2 + 2 * c]};
                yk = CR{yx, yy};
            }
        }
        const R tau = stau * stau;
        const CR w = tau * cfmac(pv, yk, sx);
        const CR v0 = l == K ? vkk : x0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const CR wc = CR{__shfl_sync(gm, w.x, c, G), __shfl_sync(gm, w.y, c, G)};
            if (l >= K) y0[K + 1 + c] = cfms(v0, wc, y0[K + 1 + c]);
            y1[K + 1 + c] = cfms(x1, wc, y1[K + 1 + c]);
        }
        U[K * 2 * G + l] = ccast<RB>(stau * v0);
        U[K * 2 * G + l + G] = ccast<RB>(stau * x1);
        if (l == K) y0[K] = CR{-pv.x, -pv.y};
        qr_steps<CHI, G, K + 1>(y0, y1, U, l, gm);
    }
}

// Back-application of NK reflectors, last first: E <- (I - u u^H) E for CHI columns, rows l and
// l + G of a lane.
template <int CHI, int G, int NK = CHI, typename RB>
__device__ __forceinline__ void apply_reflectors(C<RB> (&E0)[CHI], C<RB> (&E1)[CHI], const C<RB>* U, int l,
                                                 unsigned gm) {
    for (int k = NK - 1; k >= 0; --k) {
        const C<RB> v0 = U[k * 2 * G + l], v1 = U[k * 2 * G + l + G];
        RB s[2 * CHI];
#pragma unroll
        for (int c = 0; c < CHI; ++c) {
            const C<RB> d = cfmac(v0, E0[c], cfmac(v1, E1[c], C<RB>{(RB)0, (RB)0}));
            s[2 * c] = d.x;
            s[2 * c + 1] = d.y;
        }
        group_sums<G>(s, gm);
#pragma unroll
        for (int c = 0; c < CHI; ++c) {
            const C<RB> d = C<RB>{s[2 * c], s[2 * c + 1]};
            E0[c] = cfms(v0, d, E0[c]);
            E1[c] = cfms(v1, d, E1[c]);
        }
    }
}

// 2 log(1 - d), Eq. (gate_fidelity); the series drops terms below 1e-20
__device__ __forceinline__ double log_fidelity(double d) {
    return d < 1e-5 ? -2.0 * d * fma(d, fma(d, 1.0 / 3.0, 0.5), 1.0) : 2.0 * log1p(-d);
}

// Truncation of a core to chi (App. D "Truncation") by its first NM lanes: n2 the squared column
// norms of A = U S, perm their order (descending).  Lane r takes the r-th largest: writes lambda_e
// and isig[r] = 1 / sigma_r for the first CHI, adds the discarded weight and the log-fidelity, and
// returns the number of triplets kept.
template <int NM, int CHI, bool LOG32>
__device__ __forceinline__ int truncate_core(const double* n2, const int* perm, double* isig, double* lam_e,
                                             double* stats, int chi, double cut, int r) {
    const unsigned mk = group_mask<NM>();
    const double s2 = n2[perm[r]];
    const double is = s2 > 1e-300 ? nr_rsqrt(s2) : 0.0;
    const double sv = s2 * is;
    const double smax = __shfl_sync(mk, sv, 0, NM);
    const int cnt = __popc(__ballot_sync(mk, sv > cut * smax) & mk);
    int keep = cnt < chi ? cnt : chi;
    if (keep < 1) keep = 1;
    double kd[2] = {r < keep ? s2 : 0.0, r < keep ? 0.0 : s2};
    group_sums<NM>(kd, mk);
    const double kept = kd[0], drop = kd[1];
    const double inv = kept > 0.0 ? nr_rsqrt(kept) : 0.0;
    if (r < CHI) {
        lam_e[r] = r < keep ? sv * inv : 0.0;
        isig[r] = is;
    }
    if (r == 0) {
        const double tot = kept + drop;
        const double disc = tot > 0.0 ? drop * nr_rcp(tot) : 0.0;
        atomicAdd(&stats[0], disc);
        // log of the gate fidelity (1 - disc)^2, Eq. (gate_fidelity); a float log in the mixed mode
        atomicAdd(&stats[1], LOG32 ? 2.0 * (double)log1pf(-(float)disc) : log_fidelity(disc));
    }
    return keep;
}

// The diagonal gate phases of gates first .. first + PB - 1 of the team's sequence (colour by colour,
// every nt-th gate of a colour from gteam on), four lanes per gate: the FP64 sine and cosine (about 50
// instructions) once per PB gates instead of once per gate.
template <int CHI, class Mode>
__device__ void gate_phases(const Ctx& c, int first, int gteam, int nt, int tid, GateSm<CHI, Mode>& sm, double tZ) {
    constexpr int PB = GateSm<CHI, Mode>::PB;
    if (tid >= 4 * PB) return;
    int r = first + tid / 4, idx = -1;
    for (int col = 0; col < c.ncol && idx < 0; ++col) {
        const int beg = c.colour_off[col] + gteam, end = c.colour_off[col + 1];
        const int cnt = beg < end ? (end - beg + nt - 1) / nt : 0;
        if (r < cnt) idx = beg + r * nt;
        else r -= cnt;
    }
    if (idx < 0) return;
    const int4 a = c.gates[idx].a;
    const double ha = c.hd[a.y], hb = c.hd[a.z], Je = c.J[a.x];
    const double za = 1.0 - 2.0 * ((tid >> 1) & 1), zb = 1.0 - 2.0 * (tid & 1);
    double sn, cs;
    sincos(-tZ * (Je * za * zb + ha * za + hb * zb), &sn, &cs);
    sm.phases[tid] = cd{cs, sn};
}

template <int CHI, class Mode>
__device__ void gate_edge(const Ctx& c, const GateMeta& gm_, const cd* ph, int tid, int team, GateSm<CHI, Mode>& sm,
                          double cX, double sX, bool pre, double cXp, double sXp) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    constexpr int NM = 2 * CHI, NR = CHI * CHI, G = NR / 2, TEAM = 2 * CHI * CHI, H = CHI * CHI * CHI;
    CT* Gam = (CT*)c.Gamma;
    const int e = gm_.a.x, bits = gm_.a.w;
    const int blk = tid / G, l = tid % G, x = blk >> 1, i = blk & 1;
    const unsigned gm = group_mask<G>();
    auto stride = [](int k) { return k == 0 ? CHI * CHI : (k == 1 ? CHI : 1); };

    // ---- rows l and l + G of the lane's block, weighted with the other bonds ----
    cd y0[CHI], y1[CHI];
    double w0, w1;
    {
        const int slot = (bits >> (2 * x)) & 3, vtx = x ? gm_.a.z : gm_.a.y;
        const int e0 = x ? gm_.b.z : gm_.b.x, e1 = x ? gm_.b.w : gm_.b.y;
        int o0, o1;
        others_of(slot, o0, o1);
        const int ss = stride(slot), s0 = stride(o0), s1 = stride(o1);
        const CT* g = Gam + (size_t)vtx * (2 * H) + l / CHI * s0 + l % CHI * s1;
        const int d1 = G / CHI * s0;   // G is a multiple of CHI: row l + G lies G / CHI further along slot o0
        CT t0[CHI], t1[CHI];
        const bool lead = pre && ((bits >> (4 + x)) & 1);
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) {
            t0[cc] = ldcg(g + i * H + cc * ss);
            t1[cc] = ldcg(g + i * H + cc * ss + d1);
        }
        w0 = lam_get(c.lam, CHI, e0, l / CHI) * lam_get(c.lam, CHI, e1, l % CHI);
        w1 = lam_get(c.lam, CHI, e0, (l + G) / CHI) * lam_get(c.lam, CHI, e1, l % CHI);
        if (tid < CHI) sm.lab[tid] = __ldcg(c.lam + (size_t)e * CHI + tid);
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc) {
            y0[cc] = ccast<double>(t0[cc]);
            y1[cc] = ccast<double>(t1[cc]);
            if (lead) {   // the leading mixing gate [[c, -i s], [-i s, c]]
                const cd p0 = ccast<double>(ldcg(g + (i ^ 1) * H + cc * ss));
                const cd p1 = ccast<double>(ldcg(g + (i ^ 1) * H + cc * ss + d1));
                y0[cc] = cd{cXp * y0[cc].x + sXp * p0.y, cXp * y0[cc].y - sXp * p0.x};
                y1[cc] = cd{cXp * y1[cc].x + sXp * p1.y, cXp * y1[cc].y - sXp * p1.x};
            }
            y0[cc] = w0 * y0[cc];
            y1[cc] = w1 * y1[cc];
        }
        if (tid == 0) sm.nrot = 0;
        team_bar<TEAM>(team);   // lab; the previous edge's readers of sm are done
    }

    // ---- Householder QR of the four CHI^2 x CHI blocks; R (side a times lambda) goes to sm.V ----
    qr_steps<CHI, G, 0>(y0, y1, &sm.U[blk][0][0], l, gm);
    if (l < CHI) {
#pragma unroll
        for (int cc = 0; cc < CHI; ++cc)
            if (cc >= l) sm.V[(blk * CHI + l) * CHI + cc] = x == 0 ? sm.lab[cc] * y0[cc] : y0[cc];
    }
    team_bar<TEAM>(team);

    // ---- core matrix M (column-major NM x NM) ----
    for (int t = tid; t < NM * NM; t += TEAM) {
        const int col = t / NM, row = t % NM;
        const int ia = row / CHI, r = row % CHI, ib = col / CHI, rp = col % CHI;
        const cd* Ra = sm.V + (ia * CHI + r) * CHI;
        const cd* Rb = sm.V + ((2 + ib) * CHI + rp) * CHI;
        cd acc = cd{0.0, 0.0};
        const int j0 = r > rp ? r : rp;
        for (int j = j0; j < CHI; ++j) acc = cfma(Ra[j], Rb[j], acc);
        sm.M[t] = ph[2 * ia + ib] * acc;
    }
    team_bar<TEAM>(team);
    // rounding-level entries of the core (graded spectra of the early anneal) are zeroed first
    if constexpr (TEAM <= 32) prune_noise<NM>(sm.M, tid, WarpGroup{group_mask<TEAM>()});
    else prune_noise<NM>(sm.M, tid, TeamGroup<TEAM>{team, &sm.flag});

    // ---- SVD of M: an FP32 Jacobi solve brought to FP64 accuracy by refinement passes ----
    // (refined_svd; before it, FP64 mode ran 6 to 11 FP64 Jacobi sweeps, and the mixed mode one or
    // two FP64 polish sweeps)
    SvdCount done;
    auto svd = [&](const auto& grp) {
        return refined_svd<NM, !Mode::mixed>(sm.M, sm.V, sm.M32, sm.V32, sm.G, sm.sig, &sm.relmask, tid, grp,
                                             group_mask<NM>(), c.svd_cut, c.chi, Mode::mixed ? 1e-5f : 1e-8f,
                                             Mode::mixed ? 1e-12 : 1e-15);
    };
    if constexpr (TEAM <= 32) done = svd(WarpGroup{group_mask<TEAM>()});
    else done = svd(TeamGroup<TEAM>{team, &sm.flag});
    if (done.rot) atomicAdd(&sm.nrot, done.rot);
    if (tid < NM) sm.perm[desc_rank_bits(sm.sig, NM, tid)] = tid;   // sm.sig: squared column norms
    team_bar<TEAM>(team);
    if (tid < NM) {   // lane r holds the r-th largest singular value
        const int k = truncate_core<NM, CHI, Mode::mixed>(sm.sig, sm.perm, sm.isig, c.lam + (size_t)e * CHI, c.stats, c.chi,
                                                          c.svd_cut, tid);
        if (tid == 0) {
            atomicAdd(&c.stats[2], (double)done.pairs);
            atomicAdd(&c.stats[3], (double)sm.nrot);
            atomicMax(&c.ctl->gate_sw_max, done.passes);
            atomicMax(&c.ctl->gate_sw32_max, done.sweeps32);
            sm.keep = k;
        }
    }
    team_bar<TEAM>(team);
    const int keep = sm.keep;

    // ---- new Gamma: reflectors of each block applied to U (side a) / V^* (side b) ----
    // FP64 mode in double, mixed mode in float (the result is stored in complex64).
    CT E0[CHI], E1[CHI];
#pragma unroll
    for (int cc = 0; cc < CHI; ++cc) {
        E0[cc] = CT{(TS)0, (TS)0};
        E1[cc] = CT{(TS)0, (TS)0};
        if (l < CHI && cc < keep) {
            const int pc = sm.perm[cc];
            const int row = i * CHI + l;
            const cd u = (x == 0) ? sm.isig[cc] * sm.M[pc * NM + row] : conj(sm.V[pc * NM + row]);
            E0[cc] = ccast<TS>(u);
        }
    }
    apply_reflectors<CHI, G>(E0, E1, &sm.U[blk][0][0], l, gm);
    const TS iw0 = w0 > 0.0 ? (TS)(Mode::mixed ? nr_rcp1(w0) : nr_rcp(w0)) : (TS)0;
    const TS iw1 = w1 > 0.0 ? (TS)(Mode::mixed ? nr_rcp1(w1) : nr_rcp(w1)) : (TS)0;
    team_bar<TEAM>(team);   // everyone is done reading the reflectors
#pragma unroll
    for (int cc = 0; cc < CHI; ++cc) {
        sm.U[blk][cc][l] = iw0 * E0[cc];
        sm.U[blk][cc][l + G] = iw1 * E1[cc];
    }
    team_bar<TEAM>(team);
    // write back, applying the mixing gate to a vertex after its last gate of the layer
    const TS cs = (TS)cX, sn = (TS)sX;
    for (int t = tid; t < 2 * CHI * NR; t += TEAM) {
        const int xx = t / (CHI * NR), rem = t % (CHI * NR);
        const int col = rem / NR, row = rem % NR;
        const int slot = (bits >> (2 * xx)) & 3, vtx = xx ? gm_.a.z : gm_.a.y;
        int o0, o1;
        others_of(slot, o0, o1);
        CT g0 = sm.U[2 * xx][col][row];
        CT g1 = sm.U[2 * xx + 1][col][row];
        if ((bits >> (6 + xx)) & 1) {
            const CT a0 = g0, a1 = g1;
            // [[c, -i s], [-i s, c]]
            g0 = CT{cs * a0.x + sn * a1.y, cs * a0.y - sn * a1.x};
            g1 = CT{sn * a0.y + cs * a1.x, -sn * a0.x + cs * a1.y};
        }
        CT* g = Gam + (size_t)vtx * (2 * H) + col * stride(slot) + (row / CHI) * stride(o0) + (row % CHI) * stride(o1);
        g[0] = g0;
        g[H] = g1;
    }
}

// mixing gate on one vertex (used for degree-0 vertices only)
template <int CHI, class Mode>
__device__ void mixing_vertex(const Ctx& c, int a, int tid, int TEAM, double cX, double sX) {
    using TS = typename Mode::TS;
    constexpr int H = CHI * CHI * CHI;
    C<TS>* g = (C<TS>*)c.Gamma + (size_t)a * 2 * H;
    for (int r = tid; r < H; r += TEAM) {
        const C<TS> a0 = ldcg(g + r), a1 = ldcg(g + H + r);
        const TS cs = (TS)cX, sn = (TS)sX;
        g[r] = C<TS>{cs * a0.x + sn * a1.y, cs * a0.y - sn * a1.x};
        g[H + r] = C<TS>{sn * a0.y + cs * a1.x, -sn * a0.x + cs * a1.y};
    }
}

// ===========================================================================
// BP init (one warp per vertex): symmetric split, warm start, and in the mixed mode
// the FP64 contraction of the warm start F0 = F(m0, m0), kept as its trace t0 and
// the defect D0 = F0 - t0 m0 (complex64; |D0| is of the order of the corrections).
// ===========================================================================
template <int CHI, class Mode>
__device__ void bp_init_vertex(const Ctx& c, int a, int tid, int cur, bool warm, double* wsm, cd* tsm) {
    using TS = typename Mode::TS;
    constexpr int H = CHI * CHI * CHI, CC = CHI * CHI, TEAM = Shape<CHI>::TV;
    const int4 ve = c.vert_edges[a];
    const int es[3] = {ve.x, ve.y, ve.z};
    // wsm[0 .. 3CHI): lambda^{1/2} per slot; wsm[3CHI .. 6CHI): m0 diagonal per slot;
    // wsm[6CHI .. 6CHI + 3): (sum lambda)^{-1/2} per slot
    if (tid < 3 * CHI) {
        const int k = tid / CHI, j = tid % CHI;
        const double lj = lam_get(c.lam, CHI, es[k], j);
        wsm[tid] = nr_sqrt(lj);
        double s = 0.0;
        for (int q = 0; q < CHI; ++q) s += lam_get(c.lam, CHI, es[k], q);
        wsm[3 * CHI + tid] = s > 0.0 ? lj * nr_rcp(s) : 0.0;
        if (j == 0) wsm[6 * CHI + k] = s > 0.0 ? nr_rsqrt(s) : 0.0;
    }
    __syncwarp();
    const C<TS>* g = (const C<TS>*)c.Gamma + (size_t)a * 2 * H;
    C<TS>* T = (C<TS>*)c.T + (size_t)a * 2 * H;
    // mixed: tsm holds T~ = T prod_k m0_k[j_k]^{1/2} (T as stored, in FP64), so that the warm
    // start's contraction below needs no weights in its inner loop
    const double iso = Mode::mixed ? wsm[6 * CHI] * wsm[6 * CHI + 1] * wsm[6 * CHI + 2] : 0.0;
    for (int t = tid; t < 2 * H; t += TEAM) {
        const int r = t % H;
        const int j0 = r / CC, j1 = (r / CHI) % CHI, j2 = r % CHI;
        const double f = wsm[j0] * wsm[CHI + j1] * wsm[2 * CHI + j2];
        const C<TS> tv = ccast<TS>(f * ccast<double>(ldcg(g + t)));
        T[t] = tv;
        if constexpr (Mode::mixed) tsm[t] = (f * iso) * ccast<double>(tv);
    }
    int out[3];
    for (int s = 0; s < 3; ++s) out[s] = es[s] >= 0 ? 2 * es[s] + (a == c.edge_info[es[s]].x ? 0 : 1) : -1;
    if (warm) {
        for (int t = tid; t < 3 * CC; t += TEAM) {
            const int s = t / CC, r = t % CC;
            if (out[s] < 0) continue;
            const int j = r / CHI, jp = r % CHI;
            if constexpr (!Mode::mixed) ((cd*)c.msg[cur])[(size_t)out[s] * CC + r] = cd{j == jp ? wsm[3 * CHI + s * CHI + j] : 0.0, 0.0};
            else ((cf*)c.msg[cur])[(size_t)out[s] * CC + r] = cf{0.f, 0.f};
        }
    }
    if constexpr (Mode::mixed) {
        __syncwarp();
        // upper triangle (j <= j') of F0 for the 3 outgoing slots, items spread over the warp:
        //   F0_s[j][j'] = sum_{i,p,q} m0_o0[p] m0_o1[q] T[.., j@s, ..] conj(T[.., j'@s, ..])
        //              = (sum T~[.., j@s, ..] conj(T~[.., j'@s, ..])) / (m0_s[j] m0_s[j'])^{1/2},
        // and 0 where m0_s[j] or m0_s[j'] vanishes (T vanishes there too)
        constexpr int NU = CHI * (CHI + 1) / 2;
        cd* F = tsm + 2 * H;   // [3][CC]
        for (int item = tid; item < 3 * NU; item += TEAM) {
            const int s = item / NU;
            int u = item % NU, j = 0;
            while (u >= CHI - j) { u -= CHI - j; ++j; }
            const int jp = j + u;
            if (out[s] < 0) continue;
            int o0, o1;
            others_of(s, o0, o1);
            const int ss = sstride<CHI>(s), s0 = sstride<CHI>(o0), s1 = sstride<CHI>(o1);
            cd f = cd{0.0, 0.0};
            for (int p = 0; p < CHI; ++p) {
                if (wsm[o0 * CHI + p] == 0.0) continue;
                for (int q = 0; q < CHI; ++q) {
                    if (wsm[o1 * CHI + q] == 0.0) continue;
                    for (int ii = 0; ii < 2; ++ii) {
                        const int base = ii * H + p * s0 + q * s1;
                        f = cfmac(tsm[base + jp * ss], tsm[base + j * ss], f);
                    }
                }
            }
            const double d = wsm[3 * CHI + s * CHI + j] * wsm[3 * CHI + s * CHI + jp];
            f = d > 0.0 ? nr_rsqrt(d) * f : cd{0.0, 0.0};
            F[s * CC + j * CHI + jp] = f;
            if (jp != j) F[s * CC + jp * CHI + j] = conj(f);
        }
        __syncwarp();
        for (int t = tid; t < 3 * CC; t += TEAM) {
            const int s = t / CC, r = t % CC;
            if (out[s] < 0) continue;
            const int j = r / CHI, jp = r % CHI;
            double t0 = 0.0;
            for (int q = 0; q < CHI; ++q) t0 += F[s * CC + q * CHI + q].x;
            const double m0 = (j == jp) ? wsm[3 * CHI + s * CHI + j] : 0.0;
            c.D0[(size_t)out[s] * CC + r] = ccast<float>(F[s * CC + r] - cd{t0 * m0, 0.0});
            if (r == 0) {
                const float h = (float)t0;
                c.t0[out[s]] = make_float4(h, 0.f, (float)(t0 - (double)h), 0.f);
            }
            if (j == jp) c.m0f[(size_t)out[s] * CHI + j] = (float)m0;
        }
    }
}

// ===========================================================================
// BP sweep for one vertex: all three outgoing messages at once (team TB).
//
// With T in its natural layout [i][j0][j1][j2] the message out of slot s is
//   F_s[j][j'] = sum T[..j@s..] conj(T[..j'@s..]) x (m_o0 (x) m_o1),        Eq. (local_consistency)
// computed as: first contractions along single slots (shared between the outgoing
// slots), second contractions per slot (Q_s), then the overlap with conj(T).  In the
// mixed mode the incoming messages are m = m0 + delta and only the delta terms are
// contracted (FP32): F_s - F_s(m0) = T x_{o0} delta x_{o1} m + m0_{o0} T x_{o1} delta.
// The per-vertex inputs that do not change during a BP run (T, the warm-start
// diagonals, D0, t0, this vertex's previous outgoing messages) are cached in the
// team's shared memory across sweeps.
// ===========================================================================
template <int CHI, class Mode, int TB>
struct BPSm {
    using TS = typename Mode::TS;
    static constexpr int H2 = 2 * CHI * CHI * CHI, CC = CHI * CHI, NP = Mode::mixed ? 3 : 2;
    // lanes that share one 2 x 2 block of an outgoing message, each summing a slice of the
    // 2 CHI^2 columns: the largest power of two (at most 32 and 2 CHI^2) that keeps all
    // 3 (CHI/2)^2 blocks of the three slots within the team
    static constexpr int fslices() {
        int ns = 1;
        while (2 * ns <= 32 && 2 * ns <= 2 * CC && 3 * (CHI / 2) * (CHI / 2) * 2 * ns <= TB) ns *= 2;
        return ns;
    }
    static constexpr int NS = fslices();
    // FP64 mode: the overlap stage keeps every lane busy instead (FP64 instructions cost per
    // warp, so the fewer per lane the better): NPART lanes per (j, j') split the (i, u) sum
    // and meet by shuffles, or, where that does not divide, the sum in two halves over the
    // physical index i, added at use
    static constexpr int NPART = TB / CC;
    // mixed mode, two lanes per fiber of one slot: the fiber-wise front (bp_front_fibers)
    static constexpr bool FIBERS = Mode::mixed && CHI >= 4 && TB == 4 * CC;
    static constexpr int NPT = FIBERS ? CC / 8 > 4 ? 4 : 2 : 1;   // partial sums of a message
    static constexpr bool HALVES = !(TB % CC == 0 && NPART <= 32 && (2 * CHI) % NPART == 0);
    static_assert(CHI % 2 == 0 && 3 * (CHI / 2) * (CHI / 2) * NS <= TB, "BP team too small for the overlap stage");
    // T, P and Q in the natural index order [i][j0][j1][j2] with one padding element after
    // every (i, j0) plane, so that a stride along slot 0 does not map to one bank
    // (two for the fiber-wise front: pairs of elements are loaded at once)
    static constexpr int PS = CC + (FIBERS ? 2 : 1), H2P = 2 * CHI * PS;
    alignas(16) C<TS> T[H2P];
    C<TS> P[NP][H2P];    // FP64: T x0 m0, T x1 m1; mixed: T x0 d0, T x1 d1, T x2 d2
    C<TS> Q[FIBERS ? 1 : 3][FIBERS ? 2 : H2P];   // per outgoing slot
    alignas(16) C<TS> min[3][CC];   // incoming messages (mixed: m0 + delta)
    alignas(16) C<TS> din[3][CC];   // mixed: incoming delta
    C<TS> F[3 * NPT][CC];   // the outgoing messages before normalisation, [partial sum][slot]
    C<TS> F1[Mode::mixed ? 1 : 3][CC];   // FP64 mode with HALVES: the i = 1 half
    C<TS> prev[3][CC];   // outgoing messages of the previous sweep
    C<TS> D[3][CC];      // new - old, for the trace norm
    cf D0f[3][CC];       // mixed: warm-start defect
    float m0f[3][CHI];   // mixed: warm-start diagonals
    cf t0h[3], t0l[3];   // mixed: traces of F0, as sums of two floats
    C<TS> trs[3];        // traces of the outgoing messages (mixed: of the correction terms)
    C<TS> itr[3];        // 1 / trace (mixed: from pairs of floats, rcp_sum32)
    TS dl[3];
    TS dsum[3];          // one instance: the team's distance summed over the rounds of a sweep
    int es[3], out_idx[3], in_idx[3];
    int cached;          // vertex held in the cache, -1 if none
    // element r of the message out of slot k
    __device__ __forceinline__ C<TS> out(int k, int r) const {
        C<TS> f = F[k][r];
        if constexpr (FIBERS) {
            if (NPT == 4 || k == 2) f = f + F[3 + k][r];
            if (NPT == 4 && k == 2) f = f + (F[6 + k][r] + F[9 + k][r]);
        } else if constexpr (!Mode::mixed && HALVES) {
            f = f + F1[k][r];
        }
        return f;
    }
};

// Trace norm (sum of singular values) of the CHI x CHI matrix A (column-major, CHI^2/2 lanes; A is
// overwritten), on lane 0.  FP64 through refined_svd with the scratch after A (trace_norm_bytes in
// all): 9 us for a 4 x 4 matrix against 22 us for FP64 Jacobi sweeps without V.  FP32 by Jacobi.
template <int CHI, typename TS>
__host__ __device__ constexpr size_t trace_norm_bytes() {
    return CHI * CHI * (sizeof(TS) == 8 ? 3 * sizeof(cd) + 2 * sizeof(cf) : sizeof(cf)) + CHI * sizeof(double);
}
template <int CHI, typename TS>
__device__ __forceinline__ TS trace_norm(C<TS>* A, int g, const WarpGroup& grp) {
    constexpr int CC = CHI * CHI;
    TS s = (TS)0;
    if constexpr (sizeof(TS) == 8) {
        cd* V = A + CC;
        cd* T = V + CC;
        cf* A32 = reinterpret_cast<cf*>(T + CC);
        double* nrm = reinterpret_cast<double*>(A32 + 2 * CC);
        grp.sync();
        prune_noise<CHI>(A, g, grp);
        // tol 1e-8: the sum of the values depends on a cosine that is left only in second order, so pairs
        // of close lengths (a traceless difference has them) need no rotation beyond that
        refined_svd<CHI, true>(A, V, A32, A32 + CC, T, nrm, nullptr, g, grp, group_mask<CHI>(), 1e-16, CHI, 1e-8f, 1e-8);
        if (g == 0)
            for (int q = 0; q < CHI; ++q) s += nr_sqrt(nrm[q]);
    } else {
        jacobi_svd<CHI, TS, WarpGroup, false, false>(A, nullptr, g, grp, group_mask<CHI>(), (TS)1e-6, 60, false, nullptr,
                                                     (TS)1e-3);
        if (g == 0)
            for (int cc = 0; cc < CHI; ++cc) {
                TS n2 = (TS)0;
                for (int r = 0; r < CHI; ++r) n2 += norm2(A[cc * CHI + r]);
                s += nr_sqrt(n2);
            }
    }
    return s;
}

// The index of vertex a's outgoing message along slot k, -1 for a phantom slot, in two dependent loads.
__device__ __forceinline__ int slot_edge(const Ctx& c, int a, int k) {
    return reinterpret_cast<const int*>(c.vert_edges + a)[k];
}
__device__ __forceinline__ int slot_out(const Ctx& c, int a, int e) {
    return e >= 0 ? 2 * e + (a == c.edge_info[e].x ? 0 : 1) : -1;
}

// Fills the team's cache for vertex a; out: its message index of slot tid (lanes 0..2).  `pre`
// receives the lane's element of the incoming messages.  Where a sweep has several rounds this runs
// in each, so everything is loaded at once, after the indices that the caller has fetched a round
// ahead, and no FP64 instruction is left in it: m0 and t0 come as the floats that the init phase
// stored.  (Formed here from lambda, by the first warp of each team, they put some 20 FP64
// instructions per vertex on two of the four sub-partitions.)
template <int CHI, class Mode, int TB>
__device__ __forceinline__ void bp_prepare(const Ctx& c, int a, int tid, int team, int cur, BPSm<CHI, Mode, TB>& sm,
                                           int out, C<typename Mode::TS>& pre) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    constexpr int TEAM = TB, CC = CHI * CHI, H2 = 2 * CHI * CHI * CHI, NT = (H2 + TEAM - 1) / TEAM;
    static_assert(3 * CC <= TEAM, "one message element per lane");
    const CT* Tg = (const CT*)c.T + (size_t)a * H2;
    CT tv[NT];
#pragma unroll
    for (int q = 0; q < NT; ++q)
        if (H2 % TEAM == 0 || tid + q * TEAM < H2) tv[q] = ldcg(Tg + tid + q * TEAM);
    team_bar<TEAM>(team);   // the team may still be reading the previous vertex's cache
    if (tid < 3) {
        sm.es[tid] = out >= 0 ? out >> 1 : -1;
        sm.out_idx[tid] = out;
        sm.in_idx[tid] = out >= 0 ? out ^ 1 : -1;
    }
    team_bar<TEAM>(team);
    const CT* src = (const CT*)c.msg[cur];
    const CT z = CT{(TS)0, (TS)0};
    CT pv = z;
    cf dv = cf{0.f, 0.f};
    float mv = 0.f;
    float4 t0 = make_float4(1.f, 0.f, 0.f, 0.f);
    const int o = tid < 3 * CC ? sm.out_idx[tid / CC] : -1;
    pre = z;
    if (o >= 0) {
        pre = ldcg(src + (size_t)(o ^ 1) * CC + tid % CC);
        pv = ldcg(src + (size_t)o * CC + tid % CC);
        if constexpr (Mode::mixed) dv = ldcg(c.D0 + (size_t)o * CC + tid % CC);
    }
    if constexpr (Mode::mixed) {
        if (tid < 3 * CHI) {
            const int om = sm.out_idx[tid / CHI];
            mv = om >= 0 ? __ldcg(c.m0f + (size_t)om * CHI + tid % CHI) : (tid % CHI == 0 ? 1.f : 0.f);
        }
        if (tid < 3 && out >= 0) t0 = __ldcg(c.t0 + out);
    }
#pragma unroll
    for (int q = 0; q < NT; ++q) {
        const int t = tid + q * TEAM;
        if (H2 % TEAM == 0 || t < H2) sm.T[t + (t / CC) * (BPSm<CHI, Mode, TB>::PS - CC)] = tv[q];
    }
    if (tid < 3 * CC) {
        sm.prev[tid / CC][tid % CC] = pv;
        if constexpr (Mode::mixed) sm.D0f[tid / CC][tid % CC] = dv;
    }
    if constexpr (Mode::mixed) {
        if (tid < 3 * CHI) sm.m0f[tid / CHI][tid % CHI] = mv;
        if (tid < 3) {
            sm.t0h[tid] = cf{t0.x, t0.y};
            sm.t0l[tid] = cf{t0.z, t0.w};
        }
    }
    if (tid == 0) sm.cached = a;
    team_bar<TEAM>(team);
}

// The contractions of a sweep, fiber by fiber (mixed mode, team of 4 CHI^2 lanes = two sets of one lane
// per fiber).  Shared-memory loads bounded the element-wise form (two loads of 8 bytes per
// complex product; at chi = 4 about 3800 of the 4400 cycles of a vertex's share of an SM).  Here a
// lane loads a fiber of T or P once, in pairs, and forms its outputs from it, the message entries
// are broadcasts to the whole warp, and a fiber of Q stays in registers until its overlap with
// conj(T) is summed: about 140 load transactions per warp and vertex instead of 480 (chi = 4).
//   P_k = T x_k delta_k: slot 0 by set 0, slot 1 by set 1, slot 2 by both (half of the outputs each);
//   Q_0 = P_1 x_2 m_2 + m0_1 P_2 (set 0), Q_1 = P_0 x_2 m_2 + m0_0 P_2 (set 1),
//   Q_2 = P_0 x_1 m_1 + m0_0 P_1 (both, half of the outputs each);
//   F_s[j][j'] = sum Q_s[.., j@s, ..] conj(T[.., j'@s, ..]).
template <int CHI>
__device__ __forceinline__ void load_fiber(const cf* p, cf (&f)[CHI]) {
#pragma unroll
    for (int q = 0; q < CHI; q += 2) {
        const float4 v = *reinterpret_cast<const float4*>(p + q);
        f[q] = cf{v.x, v.y};
        f[q + 1] = cf{v.z, v.w};
    }
}
// outputs x0 and x0 + 1 of a fiber contracted with y[q][x]
template <int CHI>
__device__ __forceinline__ void fiber_pair(const cf (&in)[CHI], const cf* y, int x0, cf& a, cf& b) {
#pragma unroll
    for (int q = 0; q < CHI; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(y + q * CHI + x0);
        a = cfma(in[q], cf{v.x, v.y}, a);
        b = cfma(in[q], cf{v.z, v.w}, b);
    }
}
// sum of ov[j'] over the CHI lanes of a fiber row (lane j' ends with ov[j']) and, where the two
// physical indices share a warp (CHI = 4), over them
template <int CHI>
__device__ __forceinline__ cf fiber_sum(cf (&ov)[CHI]) {
    float s[2 * CHI];
#pragma unroll
    for (int q = 0; q < CHI; ++q) {
        s[2 * q] = ov[q].x;
        s[2 * q + 1] = ov[q].y;
    }
    rs_level<CHI / 2, 2 * CHI>(s, 0xffffffffu, threadIdx.x & (CHI - 1));
    if constexpr (CHI == 4) {
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 16);
        s[1] += __shfl_xor_sync(0xffffffffu, s[1], 16);
    }
    return cf{s[0], s[1]};
}
template <int CHI, class Mode, int TB>
__device__ __forceinline__ void bp_front_fibers(int tid, int team, BPSm<CHI, Mode, TB>& sm) {
    using SM = BPSm<CHI, Mode, TB>;
    constexpr int CC = CHI * CHI, NF = 2 * CC, S0 = SM::PS, S1 = CHI, HP = CHI * SM::PS, HALF = CHI / 2;
    const int set = tid / NF, f = tid % NF, i = f / CC, u = (f / CHI) % CHI, v = f % CHI;
    const cf z = cf{0.f, 0.f};
    {   // P_0 or P_1
        const int st = set ? S1 : S0, base = i * HP + u * (set ? S0 : S1) + v;
        cf in[CHI];
#pragma unroll
        for (int q = 0; q < CHI; ++q) in[q] = sm.T[base + q * st];
#pragma unroll
        for (int x = 0; x < CHI; x += 2) {
            cf a = z, b = z;
            fiber_pair<CHI>(in, sm.din[set], x, a, b);
            sm.P[set][base + x * st] = a;
            sm.P[set][base + (x + 1) * st] = b;
        }
    }
    {   // half of the outputs of P_2
        const int base = i * HP + u * S0 + v * S1;
        cf in[CHI];
        load_fiber<CHI>(sm.T + base, in);
#pragma unroll
        for (int x = 0; x < HALF; x += 2) {
            cf a = z, b = z;
            fiber_pair<CHI>(in, sm.din[2], set * HALF + x, a, b);
            *reinterpret_cast<float4*>(sm.P[2] + base + set * HALF + x) = float4{a.x, a.y, b.x, b.y};
        }
    }
    team_bar<TB>(team);
    const int j = u, a0 = v;   // message index and the index summed over the CHI neighbouring lanes
    if (sm.es[set] >= 0) {   // the same for the set
        // set 0: (j0, j1) = (j, a0), set 1: (a0, j)
        const int base = i * HP + (set ? a0 : j) * S0 + (set ? j : a0) * S1;
        cf in[CHI], q[CHI], p2[CHI];
        load_fiber<CHI>((set ? sm.P[0] : sm.P[1]) + base, in);
        load_fiber<CHI>(sm.P[2] + base, p2);
        const float w = set ? sm.m0f[0][a0] : sm.m0f[1][a0];
#pragma unroll
        for (int b = 0; b < CHI; ++b) q[b] = w * p2[b];
#pragma unroll
        for (int b = 0; b < CHI; b += 2) fiber_pair<CHI>(in, sm.min[2], b, q[b], q[b + 1]);
        cf ov[CHI];
        const cf* Tb = sm.T + i * HP + a0 * (set ? S0 : S1);
#pragma unroll
        for (int jp = 0; jp < CHI; ++jp) {
            cf t[CHI];
            load_fiber<CHI>(Tb + jp * (set ? S1 : S0), t);
            ov[jp] = z;
#pragma unroll
            for (int b = 0; b < CHI; ++b) ov[jp] = cfmac(t[b], q[b], ov[jp]);
        }
        const cf r = fiber_sum<CHI>(ov);
        if (CHI != 4 || i == 0) sm.F[(CHI == 4 ? 0 : 3 * i) + set][j * CHI + a0] = r;
    }
    if (sm.es[2] >= 0) {
        // j2 = j, j0 = a0, j1 = b in the set's half
        const int base = i * HP + a0 * S0 + j;
        cf in[CHI], q[HALF];
#pragma unroll
        for (int x = 0; x < CHI; ++x) in[x] = sm.P[0][base + x * S1];
        const float w = sm.m0f[0][a0];
#pragma unroll
        for (int b = 0; b < HALF; ++b) q[b] = w * sm.P[1][base + (set * HALF + b) * S1];
#pragma unroll
        for (int b = 0; b < HALF; b += 2) fiber_pair<CHI>(in, sm.min[1], set * HALF + b, q[b], q[b + 1]);
        cf ov[CHI];
#pragma unroll
        for (int jp = 0; jp < CHI; ++jp) ov[jp] = z;
#pragma unroll
        for (int b = 0; b < HALF; ++b) {
            cf t[CHI];
            load_fiber<CHI>(sm.T + i * HP + a0 * S0 + (set * HALF + b) * S1, t);
#pragma unroll
            for (int jp = 0; jp < CHI; ++jp) ov[jp] = cfmac(t[jp], q[b], ov[jp]);
        }
        const cf r = fiber_sum<CHI>(ov);
        if (CHI != 4 || i == 0) sm.F[3 * (CHI == 4 ? set : i + 2 * set) + 2][j * CHI + a0] = r;
    }
    team_bar<TB>(team);
}

// The warp of a team that takes a stage of one warp's work: those of a block's teams spread over the
// sub-partitions (a team of two warps has two of them, every other team the same two).
template <int TEAM>
__device__ __forceinline__ int lone_warp(int team) {
    return TEAM == 64 ? (team >> 1) & 1 : team % (TEAM / 32);
}

// The contractions of a sweep element by element (FP64 mode, and the shapes without a fiber-wise form).
// lone: no block has a second vertex.
template <int CHI, class Mode, int TB>
__device__ __forceinline__ void bp_front_elements(int tid, int team, bool lone, BPSm<CHI, Mode, TB>& sm) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    using SM = BPSm<CHI, Mode, TB>;
    constexpr int TEAM = TB, CC = CHI * CHI, H = CHI * CHI * CHI, H2 = 2 * H;
    // strides in the padded shared-memory layout: slot 0, slot 1 (slot 2 has stride 1), i
    constexpr int S0 = SM::PS, S1 = CHI, HP = CHI * SM::PS;
    const CT z = CT{(TS)0, (TS)0};
    constexpr bool EVEN = H2 % TEAM == 0;   // whole tensors per team pass: slots fixed at compile time
    auto slot_stride = [](int k) { return k == 0 ? S0 : (k == 1 ? S1 : 1); };
    // a stage of no more than one warp's work: the teams of a block take warps on different sub-partitions
    const int wt = (tid + TEAM - 32 * lone_warp<TEAM>(team)) % TEAM;
    if constexpr (!Mode::mixed) {
        // the messages on the slots before s contracted into T, those after s (as m^H) into the other
        // factor of the overlap: L_1 = T x_0 m_0, R_1 = T x_2 m_2^H, L_2 = L_1 x_1 m_1, R_0 = R_1 x_1 m_1^H;
        // F_0 = <T, R_0>, F_1 = <L_1, R_1>, F_2 = <L_2, T>: seven tensor-sized products instead of
        // the eight of two first and three second contractions
        auto contract = [&](const CT* src, CT* dst, int k, bool adj, int e) {
            const int pe = e + e / CC, st = slot_stride(k);
            const int x = k == 0 ? (e / CC) % CHI : (k == 1 ? (e / CHI) % CHI : e % CHI);
            const int base = pe - x * st;
            const CT* y = sm.min[k];
            CT acc = z;
#pragma unroll
            for (int q = 0; q < CHI; ++q)
                acc = adj ? cfmac(y[x * CHI + q], src[base + q * st], acc) : cfma(src[base + q * st], y[q * CHI + x], acc);
            dst[pe] = acc;
        };
        auto both = [&](const CT* s0, CT* d0, int k0, const CT* s1, CT* d1, int k1) {
            if constexpr (EVEN) {
#pragma unroll
                for (int w = 0; w < H2 / TEAM; ++w) contract(s0, d0, k0, false, tid + w * TEAM);
#pragma unroll
                for (int w = 0; w < H2 / TEAM; ++w) contract(s1, d1, k1, true, tid + w * TEAM);
            } else {
                // CHI = 2, 16 elements each.  As two branches of one warp the contractions would be issued
                // one after the other.  Where a block has several vertices they fill one warp in one
                // instruction stream (m or m^H by index and sign: half the FP64 instructions), for
                // a lone vertex two warps (no selects: 7.5 -> 7.4 us per sweep at n = 100).
                static_assert(H2 == 16 && TEAM >= 64, "two contractions in one warp, or in two");
                auto one = [&](const CT* src, CT* dst, int k, bool adj, int e) {
                    const int pe = e + e / CC, st = slot_stride(k);
                    const int x = k == 0 ? (e / CC) % CHI : (k == 1 ? (e / CHI) % CHI : e % CHI);
                    const int base = pe - x * st;
                    CT acc = z;
#pragma unroll
                    for (int q = 0; q < CHI; ++q) {
                        CT m = sm.min[k][adj ? x * CHI + q : q * CHI + x];
                        if (adj) m.y = __longlong_as_double(__double_as_longlong(m.y) ^ LLONG_MIN);
                        acc = cfma(m, src[base + q * st], acc);
                    }
                    dst[pe] = acc;
                };
                if (lone) {
                    if (tid < H2) one(s0, d0, k0, false, tid);
                    else if (tid >= 32 && tid < 32 + H2) one(s1, d1, k1, true, tid - 32);
                } else if (wt < 2 * H2) {
                    const bool adj = wt >= H2;
                    one(adj ? s1 : s0, adj ? d1 : d0, adj ? k1 : k0, adj, wt % H2);
                }
            }
            team_bar<TEAM>(team);
        };
        both(sm.T, sm.P[0], 0, sm.T, sm.P[1], 2);
        both(sm.P[0], sm.Q[0], 1, sm.P[1], sm.Q[1], 1);
    } else {
        // first contractions along one slot: P_k[.., x@k, ..] = sum_q T[.., q@k, ..] y_k[q][x]
        //   FP64: y = m (k = 0, 1); mixed: y = delta (k = 0, 1, 2)
        constexpr int NP = SM::NP;
        // e: natural index of an element, pe: its padded position
        auto p_elem = [&](int k, int e) {
            const int pe = e + e / CC;
            const int st = slot_stride(k);
            const int x = k == 0 ? (e / CC) % CHI : (k == 1 ? (e / CHI) % CHI : e % CHI);
            const int base = pe - x * st;
            const CT* y = Mode::mixed ? sm.din[k] : sm.min[k];
            CT acc = z;
#pragma unroll
            for (int q = 0; q < CHI; ++q) acc = cfma(sm.T[base + q * st], y[q * CHI + x], acc);
            sm.P[k][pe] = acc;
        };
        if constexpr (EVEN) {
#pragma unroll
            for (int k = 0; k < NP; ++k)
#pragma unroll
                for (int w = 0; w < H2 / TEAM; ++w) p_elem(k, tid + w * TEAM);
        } else {
            for (int t = tid; t < NP * H2; t += TEAM) p_elem(t / H2, t % H2);
        }
        team_bar<TEAM>(team);
        // second contractions per outgoing slot s (natural layout, slot-s index = j):
        //   Q_0[i][j][a][b] = sum_q P_1[i][j][a][q] m_2[q][b]  (+ m0_1[a] P_2[i][j][a][b])
        //   Q_1[i][a][j][b] = sum_q P_0[i][a][j][q] m_2[q][b]  (+ m0_0[a] P_2[i][a][j][b])
        //   Q_2[i][a][b][j] = sum_q P_0[i][a][q][j] m_1[q][b]  (+ m0_0[a] P_1[i][a][b][j])
        auto q_elem = [&](int s, int e) {
            const int pe = e + e / CC;
            const int j0 = (e / CC) % CHI, j1 = (e / CHI) % CHI, j2 = e % CHI;
            CT acc = z;
            if (s == 2) {
#pragma unroll
                for (int q = 0; q < CHI; ++q) acc = cfma(sm.P[0][pe - j1 * S1 + q * S1], sm.min[1][q * CHI + j1], acc);
            } else {
                const CT* Ps = (s == 0) ? sm.P[1] : sm.P[0];
#pragma unroll
                for (int q = 0; q < CHI; ++q) acc = cfma(Ps[pe - j2 + q], sm.min[2][q * CHI + j2], acc);
            }
            if constexpr (Mode::mixed) {
                const float w = (s == 0) ? sm.m0f[1][j1] : sm.m0f[0][j0];
                const CT pv = (s == 2) ? sm.P[1][pe] : sm.P[2][pe];
                acc = acc + w * pv;
            }
            sm.Q[s][pe] = acc;
        };
        if constexpr (EVEN) {
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                if (sm.es[s] < 0) continue;
#pragma unroll
                for (int w = 0; w < H2 / TEAM; ++w) q_elem(s, tid + w * TEAM);
            }
        } else {
            for (int t = tid; t < 3 * H2; t += TEAM) {
                const int s = t / H2;
                if (sm.es[s] >= 0) q_elem(s, t % H2);
            }
        }
        team_bar<TEAM>(team);
    }
    // overlaps with conj(T): F_s[j][j'] = sum over the 2 CHI^2 columns (i, u@o0, v@o1) of
    // Q_s[.., j@s, ..] conj(T[.., j'@s, ..]).  Mixed mode: a lane holds a 2 x 2 block of
    // (j, j') over a slice of the columns, so that every element it loads feeds two products;
    // the NS lanes of a block then sum by shuffles.
    if constexpr (Mode::mixed) {
        constexpr int NBJ = CHI / 2, NB = NBJ * NBJ, K = 2 * CC, NS = SM::NS, CPL = K / NS;
        if (tid < 3 * NB * NS) {
            const int s = tid / (NB * NS), rem = tid % (NB * NS);
            const int b = rem / NS, slice = rem % NS;
            const int j0 = 2 * (b / NBJ), jp0 = 2 * (b % NBJ);
            if (sm.es[s] >= 0) {   // the same for the NS lanes of a block
                const int ss = slot_stride(s);
                const int so = s == 0 ? S1 : S0, st2 = s == 2 ? S1 : 1;   // strides of the two other slots
                const CT* Qs = sm.Q[s];
                CT a00 = z, a01 = z, a10 = z, a11 = z;
#pragma unroll
                for (int w = 0; w < CPL; ++w) {
                    const int cl = slice * CPL + w;
                    const int off = (cl / CC) * HP + ((cl / CHI) % CHI) * so + (cl % CHI) * st2;
                    const CT q0 = Qs[off + j0 * ss], q1 = Qs[off + (j0 + 1) * ss];
                    const CT t0 = sm.T[off + jp0 * ss], t1 = sm.T[off + (jp0 + 1) * ss];
                    a00 = cfmac(t0, q0, a00);
                    a01 = cfmac(t1, q0, a01);
                    a10 = cfmac(t0, q1, a10);
                    a11 = cfmac(t1, q1, a11);
                }
                const unsigned gm = group_mask<NS>();
                a00.x = group_sum<NS>(a00.x, gm);
                a00.y = group_sum<NS>(a00.y, gm);
                a01.x = group_sum<NS>(a01.x, gm);
                a01.y = group_sum<NS>(a01.y, gm);
                a10.x = group_sum<NS>(a10.x, gm);
                a10.y = group_sum<NS>(a10.y, gm);
                a11.x = group_sum<NS>(a11.x, gm);
                a11.y = group_sum<NS>(a11.y, gm);
                if (slice == 0) {
                    sm.F[s][j0 * CHI + jp0] = a00;
                    sm.F[s][j0 * CHI + jp0 + 1] = a01;
                    sm.F[s][(j0 + 1) * CHI + jp0] = a10;
                    sm.F[s][(j0 + 1) * CHI + jp0 + 1] = a11;
                }
            }
        }
    } else if constexpr (SM::HALVES) {
        for (int t = wt; t < 2 * 3 * CC; t += TEAM) {
            const int i = t / (3 * CC), rem = t % (3 * CC);
            const int s = rem / CC, r = rem % CC;
            if (sm.es[s] < 0) continue;
            const int j = r / CHI, jp = r % CHI;
            const int ss = slot_stride(s);
            const int so = s == 0 ? S1 : S0, st2 = s == 2 ? S1 : 1;   // strides of the two other slots
            const CT* X = s == 0 ? sm.T : (s == 1 ? sm.P[0] : sm.Q[0]);
            const CT* Y = s == 0 ? sm.Q[1] : (s == 1 ? sm.P[1] : sm.T);
            CT acc = z;
#pragma unroll
            for (int u = 0; u < CHI; ++u)
#pragma unroll
                for (int v = 0; v < CHI; ++v) {
                    const int off = i * HP + u * so + v * st2;
                    acc = cfmac(Y[off + jp * ss], X[off + j * ss], acc);
                }
            if (i == 0) sm.F[s][r] = acc;
            else sm.F1[s][r] = acc;
        }
    } else {
        constexpr int NPART = SM::NPART, PER = 2 * CHI / NPART;
        const int r = tid / NPART, part = tid % NPART;
        const int j = r / CHI, jp = r % CHI;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            if (sm.es[s] < 0) continue;
            const int ss = slot_stride(s);
            const int so = s == 0 ? S1 : S0, st2 = s == 2 ? S1 : 1;
            const CT* X = s == 0 ? sm.T : (s == 1 ? sm.P[0] : sm.Q[0]);
            const CT* Y = s == 0 ? sm.Q[1] : (s == 1 ? sm.P[1] : sm.T);
            CT acc = z;
#pragma unroll
            for (int h = 0; h < PER; ++h) {
                const int cmb = part * PER + h, i = cmb / CHI, u = cmb % CHI;
#pragma unroll
                for (int v = 0; v < CHI; ++v) {
                    const int off = i * HP + u * so + v * st2;
                    acc = cfmac(Y[off + jp * ss], X[off + j * ss], acc);
                }
            }
            acc.x = group_sum<NPART>(acc.x, group_mask<NPART>());
            acc.y = group_sum<NPART>(acc.y, group_mask<NPART>());
            if (part == 0) sm.F[s][r] = acc;
        }
    }
    team_bar<TEAM>(team);
}

// 1 / (t + d) for a complex t held as hi + lo: sums, products and the reciprocal carried as pairs of
// floats (relative error about 1e-13) and rounded to FP32 once, so that the result is the FP32
// rounding of the FP64 one.  In FP64 the same took one warp of the block 0.4 us per sweep (14
// instructions of 64 cycles) between two block barriers.
__device__ __forceinline__ void sum32(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
__device__ __forceinline__ cf rcp_sum32(cf hi, cf lo, cf d) {
    float x, xl, y, yl, h, e;
    sum32(hi.x, d.x, h, e);
    sum32(h, e + lo.x, x, xl);
    sum32(hi.y, d.y, h, e);
    sum32(h, e + lo.y, y, yl);
    if (x == 0.f && y == 0.f) return cf{0.f, 0.f};
    // scaled by a power of two to between 1 and 4, so that the squares stay in range for every trace
    // that complex64 holds (a vertex tensor may carry any factor)
    const int ex = max(__float_as_int(x) & 0x7f800000, __float_as_int(y) & 0x7f800000);
    const float sc = __int_as_float(min(max(0x7f000000 - ex, 0x00800000), 0x7e800000));
    x *= sc;
    xl *= sc;
    y *= sc;
    yl *= sc;
    const float px = __fmul_rn(x, x), py = __fmul_rn(y, y);
    float n, nl;
    sum32(px, py, n, nl);
    nl += (fmaf(x, x, -px) + 2.f * x * xl) + (fmaf(y, y, -py) + 2.f * y * yl);
    const float r = __frcp_rn(n), rl = r * (fmaf(-n, r, 1.f) - nl * r);   // r + rl = 1 / (n + nl)
    const float ax = __fmul_rn(x, r), ay = __fmul_rn(y, r);
    return cf{sc * (ax + (fmaf(x, r, -ax) + (x * rl + xl * r))), -sc * (ay + (fmaf(y, r, -ay) + (y * rl + yl * r)))};
}

// First part of the sweep for vertex a: incoming messages, the contractions, and the
// traces of the three outgoing messages with their reciprocals (left in sm.trs and sm.itr).  Only the
// team's shared memory is written.  out: as in bp_prepare, read only where the cache holds another vertex.
template <int CHI, class Mode, int TB>
__device__ void bp_front(const Ctx& c, int a, int tid, int team, int cur, BPSm<CHI, Mode, TB>& sm, bool have_pre,
                         C<typename Mode::TS> pre, int out) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    using SM = BPSm<CHI, Mode, TB>;
    constexpr int TEAM = TB, CC = CHI * CHI;
    if (sm.cached != a) {
        bp_prepare<CHI, Mode, TB>(c, a, tid, team, cur, sm, out, pre);
        have_pre = true;
    }
    const CT* src = (const CT*)c.msg[cur];
    const CT z = CT{(TS)0, (TS)0};
    // incoming messages (prefetched into `pre` by the caller when have_pre)
    for (int t = tid; t < 3 * CC; t += TEAM) {
        const int k = t / CC, r = t % CC;
        const int in = sm.in_idx[k];
        const CT lv = in >= 0 ? (have_pre ? pre : ldcg(src + (size_t)in * CC + r)) : z;
        if constexpr (!Mode::mixed) {
            sm.min[k][r] = in >= 0 ? lv : CT{(TS)(r == 0 ? 1 : 0), (TS)0};
        } else {
            const int j = r / CHI, jp = r % CHI;
            const CT dv = lv;
            sm.din[k][r] = dv;
            sm.min[k][r] = CT{dv.x + ((j == jp) ? sm.m0f[k][j] : 0.f), dv.y};
        }
    }
    team_bar<TEAM>(team);
    if constexpr (SM::FIBERS) {
        bp_front_fibers<CHI, Mode, TB>(tid, team, sm);
    } else {
        bp_front_elements<CHI, Mode, TB>(tid, team, c.n <= c.nblocks, sm);
    }
    // traces of the outgoing messages and their reciprocals (reading R10: messages are divided by
    // their complex trace).  In FP64 some 20 instructions of one warp
    const int k = Mode::mixed ? tid : tid - 32 * lone_warp<TEAM>(team);
    if (k >= 0 && k < 3) {
        CT trs = z;
#pragma unroll
        for (int j = 0; j < CHI; ++j) trs = trs + sm.out(k, j * CHI + j);
        sm.trs[k] = trs;
        if constexpr (Mode::mixed) {
            sm.itr[k] = rcp_sum32(sm.t0h[k], sm.t0l[k], trs);
        } else {
            const double n2 = norm2(trs);
            const double in2 = n2 > 0.0 ? nr_rcp(n2) : 0.0;
            sm.itr[k] = cd{trs.x * in2, -trs.y * in2};
        }
    }
    team_bar<TEAM>(team);
}

// Second part: new messages m' = F / tr F (mixed: delta' = (D0 + Fd - m0 tr Fd) / (t0 + tr Fd))
// and the distance of App. B, added to *dacc.
template <int CHI, class Mode, int TB>
__device__ void bp_back(const Ctx& c, int tid, int team, int cur, bool exact, BPSm<CHI, Mode, TB>& sm,
                        double* gacc) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    constexpr int TEAM = TB, CC = CHI * CHI;
    CT* dst = (CT*)c.msg[cur ^ 1];
    const CT z = CT{(TS)0, (TS)0};
    constexpr int GJ = CC / 2;
    constexpr bool FAST = CC <= 32;   // the elements of one message lie in one warp
    static_assert(3 * GJ <= TEAM && 3 * CHI <= 32 && 3 * CC <= TEAM, "BP team too small");
    TS f2 = (TS)0;
    if (tid < 3 * CC) {
        const int k = tid / CC, r = tid % CC;
        const int out = sm.out_idx[k];
        CT d = z;
        if (out >= 0) {
            const CT itr = sm.itr[k];
            const CT f = sm.out(k, r);
            CT num = f;
            if constexpr (Mode::mixed) {
                const int j = r / CHI, jp = r % CHI;
                num = sm.D0f[k][r] + f;
                if (j == jp) num = num - sm.m0f[k][j] * sm.trs[k];
            }
            const CT nv = itr * num;
            dst[(size_t)out * CC + r] = nv;
            d = nv - sm.prev[k][r];
            sm.prev[k][r] = nv;
        }
        if (FAST && !exact) f2 = norm2(d);
        else sm.D[k][r] = d;
    }
    // distance of App. B: trace norms ||m_new - m_old||_1 (sum of singular values) when
    // `exact`, else the Frobenius norms, a lower bound that suffices to continue
    if constexpr (FAST) {
        if (!exact) {
            if (tid < 3 * CC) {
                f2 = group_sum<CC>(f2, group_mask<CC>());
                if (tid % CC == 0) {
                    const TS f = sm.out_idx[tid / CC] >= 0 ? nr_sqrt(f2) : (TS)0;
                    if (gacc) atomicAdd(gacc, (double)f);
                    else sm.dsum[tid / CC] += f;
                }
            }
            return;
        }
    }
    team_bar<TEAM>(team);
    if (!exact) {
        if (tid < 32) {
            TS c2 = (TS)0;
            if (tid < 3 * CHI) {
                const int k = tid / CHI, cc = tid % CHI;
#pragma unroll
                for (int r = 0; r < CHI; ++r) c2 += norm2(sm.D[k][cc * CHI + r]);
            }
#pragma unroll
            for (int o = 1; o < CHI; o <<= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
            if (tid < 3 * CHI && tid % CHI == 0) sm.dl[tid / CHI] = nr_sqrt(c2);
        }
    } else if (tid < 3 * GJ) {
        const int k = tid / GJ, g = tid % GJ;
        WarpGroup grp{group_mask<GJ>()};
        CT* A = sm.D[k];
        if constexpr (!Mode::mixed) {   // with its scratch in P and Q, which are free here
            static_assert(3 * trace_norm_bytes<CHI, TS>() <= sizeof(sm.P) + sizeof(sm.Q), "scratch of the trace norms");
            A = reinterpret_cast<CT*>(reinterpret_cast<unsigned char*>(sm.P) + k * trace_norm_bytes<CHI, TS>());
            for (int r = g; r < CC; r += GJ) A[r] = sm.D[k][r];
        }
        const TS sacc = trace_norm<CHI, TS>(A, g, grp);
        if (g == 0) sm.dl[k] = sacc;
    }
    team_bar<TEAM>(team);
    if (gacc) {
        if (tid == 0) atomicAdd(gacc, (double)sm.dl[0] + (double)sm.dl[1] + (double)sm.dl[2]);
    } else if (tid < 3) {
        sm.dsum[tid] += sm.dl[tid];
    }
}

// copy a frozen instance's outgoing messages to the other buffer
template <int CHI, class Mode>
__device__ void bp_copy_vertex(const Ctx& c, int a, int tid, int TEAM, int cur) {
    using CT = C<typename Mode::TS>;
    constexpr int CC = CHI * CHI;
    const int4 ve = c.vert_edges[a];
    const int es[3] = {ve.x, ve.y, ve.z};
    const CT* src = (const CT*)c.msg[cur];
    CT* dst = (CT*)c.msg[cur ^ 1];
    for (int k = 0; k < 3; ++k) {
        if (es[k] < 0) continue;
        const int u = c.edge_info[es[k]].x;
        const int out = 2 * es[k] + (a == u ? 0 : 1);
        for (int r = tid; r < CC; r += TEAM) dst[(size_t)out * CC + r] = ldcg(src + (size_t)out * CC + r);
    }
}

// Exact distance of the sweep that wrote msg[cur_new] for the instances with need[b]
// set: trace norms of new - old for every directed message, one group of CHI^2/2
// threads per message (whole block, after a grid barrier).  Accumulates into ex[b].
template <int CHI, class Mode, int TPB, int TB>
__device__ void bp_exact_pass(const Ctx& c, int cur_new, const int* need, BPSm<CHI, Mode, TB>& sm, double* bacc,
                              double* ex) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    // the groups of a team have their matrices and scratch in its P and Q buffers
    constexpr int CC = CHI * CHI, GJ = CC / 2, FIT = (int)((sizeof(sm.P) + sizeof(sm.Q)) / trace_norm_bytes<CHI, TS>());
    constexpr int NGT = TB / GJ < FIT ? TB / GJ : FIT, TEAMS = TPB / TB;
    static_assert(NGT >= 1, "scratch of the trace norms");
    const int team = threadIdx.x / TB, gi = (threadIdx.x % TB) / GJ, g = threadIdx.x % GJ;
    CT* Dm = reinterpret_cast<CT*>(reinterpret_cast<unsigned char*>(sm.P) + (gi < NGT ? gi : 0) * trace_norm_bytes<CHI, TS>());
    const CT* nw = (const CT*)c.msg[cur_new];
    const CT* od = (const CT*)c.msg[cur_new ^ 1];
    if (threadIdx.x == 0) *bacc = 0.0;
    __syncthreads();
    const WarpGroup grp{group_mask<GJ>()};
    double mine = 0.0;
    // consecutive messages go to different blocks, then to different teams
    for (int mi = (gi * TEAMS + team) * c.nblocks + blockIdx.x; gi < NGT && mi < 2 * c.m; mi += c.nblocks * TEAMS * NGT) {
        const int inst = c.vert_inst[c.edge_info[mi >> 1].x];
        if (!need[inst]) continue;
        for (int r = g; r < CC; r += GJ) Dm[r] = ldcg(nw + (size_t)mi * CC + r) - ldcg(od + (size_t)mi * CC + r);
        const TS sacc = trace_norm<CHI, TS>(Dm, g, grp);
        if (g == 0) {
            if (c.B == 1) mine += (double)sacc;
            else atomicAdd(ex + inst, (double)sacc);
        }
        grp.sync();
    }
    if (c.B == 1) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
        if ((threadIdx.x & 31) == 0 && mine != 0.0) atomicAdd(bacc, mine);
        __syncthreads();
        if (threadIdx.x == 0 && *bacc != 0.0) atomicAdd(ex, *bacc);
    }
}

// ===========================================================================
// regauge, edge part: FP64 eigen/SVD, transforms X_a, X_b and lambda
//
// A team is CHI^2 lanes, half of them per message, or CHI^2 / 2 lanes that take the two messages in
// turn.  The three decompositions of an edge are the FP64 work: the wide team finishes an edge
// sooner (two in turn instead of three) but leaves half of its lanes idle in the third one, and the
// FP64 pipe charges a warp, not its lanes.  The narrow team runs once a sub-partition has more than
// four wide warps' worth of edges (m > SMs x 512 / CHI^2): at 10 edges per block (n = 1000, chi = 4)
// it is 9 us slower per regauge, at 165 (32 instances) a regauge is 15 % faster.
// ===========================================================================
template <int CHI>
struct RGSm {
    cd Am[2][CHI * CHI];
    cd Vm[2][CHI * CHI];
    double w[2][CHI];
    double wq[2][CHI], wiq[2][CHI];   // w^{1/2} and w^{-1/2} of the kept eigenvalues, else 0
    cd Y[2][CHI * CHI];               // scaled singular vectors of M
    cd M[CHI * CHI];
    cd VM[CHI * CHI];
    double sig[CHI];
    double isig[CHI];   // 1 / sig (0 for a zero singular value)
    int perm[CHI];
    double scal[2];
    // scratch of the decompositions
    cf A32[2][CHI * CHI];
    cf V32[2][CHI * CHI];
    cd T1[2][CHI * CHI];
    double nrm[2][CHI];
};

template <int CHI, class Mode, int TEAM>
__device__ void regauge_edge(const Ctx& c, int e, int tid, int team, int cur, RGSm<CHI>& sm) {
    constexpr int CC = CHI * CHI, GJ = CC / 2;
    static_assert(TEAM == CC || TEAM == GJ, "one or both messages at a time");
    // Hermitian parts of m_{a->b} (x = 0) and m_{b->a} (x = 1), column-major
    for (int t = tid; t < 2 * CC; t += TEAM) {
        const int x = t / CC, r = t % CC;
        const int row = r % CHI, col = r / CHI;
        cd v, vt;
        if constexpr (!Mode::mixed) {
            const cd* mm = (const cd*)c.msg[cur] + (size_t)(2 * e + x) * CC;
            v = ldcg(mm + row * CHI + col);
            vt = ldcg(mm + col * CHI + row);
        } else {
            const cf* mm = (const cf*)c.msg[cur] + (size_t)(2 * e + x) * CC;
            v = ccast<double>(ldcg(mm + row * CHI + col));
            vt = ccast<double>(ldcg(mm + col * CHI + row));
            if (row == col) {
                double s = 0.0;
                for (int q = 0; q < CHI; ++q) s += __ldcg(c.lam + (size_t)e * CHI + q);
                const double m0 = s > 0.0 ? __ldcg(c.lam + (size_t)e * CHI + row) * nr_rcp(s) : 0.0;
                v.x += m0;
                vt.x += m0;
            }
        }
        sm.Am[x][col * CHI + row] = cd{0.5 * (v.x + vt.x), 0.5 * (v.y - vt.y)};
    }
    team_bar<TEAM>(team);
    {
        // FP64 eigen-decompositions of the two Hermitian messages (the singular values of a
        // Hermitian matrix are the moduli of its eigenvalues)
        const int g = tid % GJ;
        WarpGroup grp{group_mask<GJ>()};
#pragma unroll 1
        for (int x = tid / GJ; x < 2; x += TEAM / GJ) {
            prune_noise<CHI>(sm.Am[x], g, grp);
            const SvdCount cnt = refined_svd<CHI, !Mode::mixed>(
                sm.Am[x], sm.Vm[x], sm.A32[x], sm.V32[x], sm.T1[x], sm.nrm[x], nullptr, g, grp, group_mask<CHI>(), c.eig_cut,
                CHI, Mode::mixed ? 3e-7f : 1e-8f, Mode::mixed ? 1e-13 : 1e-15);
            if (g == 0) {
                atomicAdd(&c.stats[4], (double)cnt.passes);
                atomicMax(&c.ctl->reg_sw_max, cnt.passes);
                atomicMax(&c.ctl->reg_sw32_max, cnt.sweeps32);
            }
        }
    }
    team_bar<TEAM>(team);
    for (int t = tid; t < 2 * CHI; t += TEAM) {
        const int x = t / CHI, k = t % CHI;
        double n2 = 0.0, sg = 0.0;
        for (int r = 0; r < CHI; ++r) {
            const cd av = sm.Am[x][k * CHI + r], vv = sm.Vm[x][k * CHI + r];
            n2 += norm2(av);
            sg += vv.x * av.x + vv.y * av.y;
        }
        const double wv = nr_sqrt(n2);
        sm.w[x][k] = sg >= 0.0 ? wv : -wv;
    }
    team_bar<TEAM>(team);
    // the roots of each eigenvalue once (eigenvalues at or below the cut-off count as zero)
    for (int t = tid; t < 2 * CHI; t += TEAM) {
        const int x = t / CHI, k = t % CHI;
        double wmax = 0.0;
        for (int q = 0; q < CHI; ++q) wmax = fmax(wmax, sm.w[x][q]);
        const double wk = sm.w[x][k];
        const bool kept = wk > c.eig_cut * wmax;
        const double isq = kept ? nr_rsqrt(wk) : 0.0;
        sm.wiq[x][k] = isq;
        sm.wq[x][k] = kept ? wk * isq : 0.0;
    }
    team_bar<TEAM>(team);
    // with m_x = V_x w_x V_x^H:  M = (m_0^{1/2})^T m_1^{1/2} = conj(V_0) B V_1^H with
    // B = w_0^{1/2} (V_0^T V_1) w_1^{1/2}, so the SVD of B gives U = conj(V_0) U', V = V_1 V', and the
    // transforms are X_a = conj(V_0) w_0^{-1/2} U' ||S||^{1/2}, X_b = conj(V_1) w_1^{-1/2} conj(V') ||S||^{1/2}:
    // a third of the products that forming m^{1/2} and m^{-1/2} takes
    for (int t = tid; t < CC; t += TEAM) {
        const int k = t % CHI, l = t / CHI;
        cd acc = cd{0.0, 0.0};
        for (int j = 0; j < CHI; ++j) acc = cfma(sm.Vm[0][k * CHI + j], sm.Vm[1][l * CHI + j], acc);
        sm.M[l * CHI + k] = (sm.wq[0][k] * sm.wq[1][l]) * acc;
    }
    team_bar<TEAM>(team);
    if (tid < GJ) {
        WarpGroup grp{group_mask<GJ>()};
        prune_noise<CHI>(sm.M, tid, grp);
        const SvdCount cnt = refined_svd<CHI, !Mode::mixed>(
            sm.M, sm.VM, sm.A32[0], sm.V32[0], sm.T1[0], sm.nrm[0], nullptr, tid, grp, group_mask<CHI>(), c.svd_cut, CHI,
            Mode::mixed ? 3e-7f : 1e-8f, Mode::mixed ? 1e-13 : 1e-15);
        if (tid == 0) {
            atomicAdd(&c.stats[4], (double)cnt.passes);
            atomicMax(&c.ctl->reg_sw_max, cnt.passes);
            atomicMax(&c.ctl->reg_sw32_max, cnt.sweeps32);
        }
    }
    team_bar<TEAM>(team);
    for (int cc = tid; cc < CHI; cc += TEAM) {
        double n2 = 0.0;
        for (int r = 0; r < CHI; ++r) n2 += norm2(sm.M[cc * CHI + r]);
        const double sv = nr_sqrt(n2);
        sm.sig[cc] = sv;
        sm.isig[cc] = sv > 0.0 ? nr_rcp(sv) : 0.0;
    }
    team_bar<TEAM>(team);
    for (int cc = tid; cc < CHI; cc += TEAM) sm.perm[desc_rank(sm.sig, CHI, cc)] = cc;
    team_bar<TEAM>(team);
    if (tid == 0) {
        double tot = 0.0;
        for (int cc = 0; cc < CHI; ++cc) tot += sm.sig[cc] * sm.sig[cc];
        const double nrm = nr_sqrt(tot);
        sm.scal[0] = nrm;
        sm.scal[1] = nr_sqrt(nrm);
        const double inrm = nrm > 0.0 ? nr_rcp(nrm) : 0.0;
        const double smax = sm.sig[sm.perm[0]];
        for (int r = 0; r < CHI; ++r) {
            const double s = sm.sig[sm.perm[r]];
            c.lam[(size_t)e * CHI + r] = (nrm > 0.0 && s > c.svd_cut * smax) ? s * inrm : 0.0;
        }
    }
    team_bar<TEAM>(team);
    // w_x^{-1/2} U' ||S||^{1/2} (x = 0) and w_x^{-1/2} conj(V') ||S||^{1/2} (x = 1), [column][row]; 0 beyond
    // the kept singular values
    for (int t = tid; t < 2 * CC; t += TEAM) {
        const int x = t / CC, r = t % CC, j = r / CHI, k = r % CHI;
        const int pc = sm.perm[j];
        const bool kept = sm.scal[0] > 0.0 && sm.sig[pc] > c.svd_cut * sm.sig[sm.perm[0]];
        const double f = kept ? sm.wiq[x][k] * sm.scal[1] : 0.0;
        sm.Y[x][r] = x == 0 ? (f * sm.isig[pc]) * sm.M[pc * CHI + k] : f * conj(sm.VM[pc * CHI + k]);
    }
    team_bar<TEAM>(team);
    for (int t = tid; t < 2 * CC; t += TEAM) {
        const int x = t / CC, r = t % CC, jpp = r / CHI, j = r % CHI;
        cd acc = cd{0.0, 0.0};
        for (int k = 0; k < CHI; ++k) acc = cfmac(sm.Vm[x][k * CHI + jpp], sm.Y[x][j * CHI + k], acc);
        c.X[((size_t)e * 2 + x) * CC + r] = acc;
    }
}

// regauge, vertex part: Gamma_a = T_a x_slot X (team TV, buffers in shared memory)
template <int CHI, class Mode, int TEAM>
__device__ void regauge_vertex(const Ctx& c, int a, int tid, int team, C<typename Mode::TS>* buf) {
    using TS = typename Mode::TS;
    using CT = C<TS>;
    constexpr int H = CHI * CHI * CHI, CC = CHI * CHI;
    const int4 ve = c.vert_edges[a];
    const int es[3] = {ve.x, ve.y, ve.z};
    CT* b0 = buf;
    CT* b1 = buf + 2 * H;
    CT* Xs = buf + 4 * H;   // [3][CC]
    for (int t = tid; t < 2 * H; t += TEAM) b0[t] = ldcg((const CT*)c.T + (size_t)a * 2 * H + t);
    for (int t = tid; t < 3 * CC; t += TEAM) {
        const int k = t / CC, r = t % CC;
        cd v;
        if (es[k] >= 0) {
            const int side = (c.edge_info[es[k]].x == a) ? 0 : 1;
            v = ldcg(c.X + ((size_t)es[k] * 2 + side) * CC + r);
        } else {
            v = cd{(r / CHI == r % CHI) ? 1.0 : 0.0, 0.0};
        }
        Xs[t] = ccast<TS>(v);
    }
    team_bar<TEAM>(team);
    CT* cur = b0;
    CT* nxt = b1;
    for (int k = 0; k < 3; ++k) {
        const int st = sstride<CHI>(k);
        for (int t = tid; t < 2 * H; t += TEAM) {
            const int jk = (t / st) % CHI;
            const int base = t - jk * st;
            CT acc = CT{(TS)0, (TS)0};
            for (int q = 0; q < CHI; ++q) acc = cfma(cur[base + q * st], Xs[k * CC + q * CHI + jk], acc);
            nxt[t] = acc;
        }
        team_bar<TEAM>(team);
        CT* tmp = cur;
        cur = nxt;
        nxt = tmp;
    }
    CT* g = (CT*)c.Gamma + (size_t)a * 2 * H;
    for (int t = tid; t < 2 * H; t += TEAM) g[t] = cur[t];
}

// ===========================================================================
// the persistent kernel
// ===========================================================================
template <int CHI, class Mode, unsigned PH, int V = 0>
struct SmemSize {
    using S = Shape<CHI, V>;
    static constexpr int TPB = S::TPB;
    static constexpr size_t gate = sizeof(GateSm<CHI, Mode>) * (TPB / S::TG);
    // per-team caches, block sums (64 doubles), for the teams of the shape and the wide ones
    static constexpr int WIDE_TB = !Mode::mixed && CHI == 4 && S::TB == 64 ? 128 : S::TB;
    static constexpr size_t mx(size_t a, size_t b) { return a > b ? a : b; }
    static constexpr size_t bp = mx(sizeof(BPSm<CHI, Mode, S::TB>) * (TPB / S::TB),
                                    sizeof(BPSm<CHI, Mode, WIDE_TB>) * (TPB / WIDE_TB)) + 64 * sizeof(double);
    static constexpr int rg_fit = (int)(190 * 1024 / sizeof(RGSm<CHI>));
    static constexpr int rg_teams = TPB / (S::TR / 2) < rg_fit ? TPB / (S::TR / 2) : rg_fit;   // narrow regauge teams
    static constexpr int rg_wide = TPB / S::TR < rg_fit ? TPB / S::TR : rg_fit;
    static constexpr size_t rg = sizeof(RGSm<CHI>) * rg_teams;
    static constexpr size_t rv =
        sizeof(C<typename Mode::TS>) * (4 * CHI * CHI * CHI + 3 * CHI * CHI) * (TPB / S::TRV);
    static constexpr size_t init =
        (sizeof(double) * (6 * CHI + 4) + (Mode::mixed ? sizeof(cd) * (2 * CHI * CHI * CHI + 3 * CHI * CHI) : 0)) * S::NIT;
    // bytes before the per-instance flags (which follow at this offset in the BP kernel)
    static constexpr size_t value = mx(mx((PH & PH_GATES) ? gate : 0, (PH & PH_BP) ? mx(bp, init) : 0),
                                       (PH & PH_REGAUGE) ? mx(rg, rv) : 0) + 16;
};

// The BP sweeps of one run (after bp_init_vertex) by vertex teams of TB lanes; false if a barrier gave up.
template <int CHI, class Mode, unsigned PH, int V, int TB>
__device__ __forceinline__ bool bp_sweeps(const Ctx& c, GridBarrier& gb, int& cur, unsigned char* smem) {
    using S = Shape<CHI, V>;
    const int team = threadIdx.x / TB, tid = threadIdx.x % TB;
    const int tpb_teams = S::TPB / TB;
    using CT_ = C<typename Mode::TS>;
    using SMB = BPSm<CHI, Mode, TB>;
    SMB& sm = reinterpret_cast<SMB*>(smem)[team];
    double* bsum = reinterpret_cast<double*>(smem + sizeof(SMB) * tpb_teams);
    // every block keeps its own copy of the per-instance state; all blocks take
    // identical decisions from the same accumulators, so one barrier per sweep suffices
    // (two when a sweep's lower bound falls under the threshold and the exact
    // distance is computed afterwards)
    int* done = reinterpret_cast<int*>(smem + SmemSize<CHI, Mode, PH, V>::value);
    int* exnow = done + c.B;   // this sweep computes the exact distance inline
    int* need = exnow + c.B;   // exact distance needed after the sweep
    double* thr = reinterpret_cast<double*>(smem + SmemSize<CHI, Mode, PH, V>::value +
                                            (3 * sizeof(int) * (size_t)c.B + 7) / 8 * 8);
    double* thr_hi = thr + c.B;                               // bound that lets a sweep continue
    float* thr3 = reinterpret_cast<float*>(thr_hi + c.B);     // inline-exact trigger
    const double slack = Mode::mixed ? 1e-5 : 1e-12;   // rounding of the lower bound
    for (int b = threadIdx.x; b < c.B; b += S::TPB) {
        done[b] = 0;
        exnow[b] = c.max_iter == 1;
        need[b] = 0;
        const double t = c.tol * (double)c.inst_m[b];
        thr[b] = t;
        thr_hi[b] = t / (1.0 - slack);
        thr3[b] = (float)(3.0 * t);
    }
    if (tid == 0) sm.cached = -1;   // T and D0 changed in the init phase
    if (tid < 3) sm.dsum[tid] = 0;
    __syncthreads();
    const int gteam = team * c.nblocks + blockIdx.x, nt = c.nblocks * tpb_teams;
    // the first round's instance and, in lanes 0..2, its vertex's message index; with several rounds
    // those of a vertex are fetched during the round before it
    const bool rounds = c.n > nt;
    int inst_a = gteam < c.n ? c.vert_inst[gteam] : 0;
    int out_a = gteam < c.n && tid < 3 ? slot_out(c, gteam, slot_edge(c, gteam, tid)) : -1;
    SMB* all = reinterpret_cast<SMB*>(smem);
    bool have_pre = false;
    CT_ pre = CT_{0, 0};
    int* sflag = reinterpret_cast<int*>(bsum + 48);   // [2]: need | open << 1, per sweep parity
    if (threadIdx.x == 0) sflag[0] = sflag[1] = 0;
    __syncthreads();
    // One instance: every thread takes the decision on a sweep itself, from the sum loaded right after
    // the barrier.  In the mixed mode (AHEAD) it does so only once it has formed the next sweep's
    // messages in shared memory, so that the load's latency and the decision lie behind that work
    // (n = 1000, chi = 4: 5.05 -> 4.6 us per sweep with the team-wise reciprocals); a sweep that turns
    // out not to be needed costs its first half, which is 1.9 us there but 31 us in FP64 mode, which
    // therefore decides first.  Returns -1 if a barrier gave up, 1 to stop, 0 to go on.
    constexpr bool AHEAD = Mode::mixed;
    bool ex1 = c.max_iter == 1;   // the sweep under way computes the exact distance inline
    const double thr3d = thr3[0];
    // Distances and thresholds are not negative, so their bits compare like the values (a NaN lies above
    // the infinities): every thread decides, and an FP64 comparison of 16 warps is 0.12 us of the pipe.
    auto less = [](double x, double y) { return __double_as_longlong(x) < __double_as_longlong(y); };
    auto isnan_d = [](double x) { return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL; };
    auto decide = [&](int itd, double dsum) {
        const bool last = itd + 1 >= c.max_iter;
        bool fin = false;
        if (c.inst_m[0] == 0 || isnan_d(dsum)) {
            fin = true;
        } else if (ex1) {
            fin = last || less(dsum, thr[0]);
        } else if (last || less(dsum, thr_hi[0])) {   // a bound under the threshold: the exact distance decides
            double* ex = c.acc + 3 + itd % 3;
            if (blockIdx.x == 0 && threadIdx.x == 0) ++c.ctl->exact_passes;
            if (threadIdx.x == 0) need[0] = 1;
            __syncthreads();   // the teams are done with P and Q
            bp_exact_pass<CHI, Mode, S::TPB, TB>(c, cur, need, sm, bsum + 32, ex);
            if (!grid_sync(gb, c.spin_limit)) return -1;
            dsum = __ldcg(ex);
            fin = last || less(dsum, thr[0]) || isnan_d(dsum);
            ex1 = true;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                c.inst_dist[0] = dsum;
                c.inst_iters[0] = itd + 1;
                if (fin) c.inst_done[0] = 1;
            }
            return fin ? 1 : 0;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            c.inst_dist[0] = dsum;
            c.inst_iters[0] = itd + 1;
            if (fin) c.inst_done[0] = 1;
        }
        // the next sweep is exact inline when it is the last or when this one came within a factor 3
        ex1 = itd + 2 >= c.max_iter || less(dsum, thr3d);
        return fin ? 1 : 0;
    };
    const bool one = c.B == 1;
    bool pend = false, stop = false;
    double dprev = 0.0;
    int it = 0;
    while (it < c.max_iter) {
        double* acc = c.acc + (size_t)(it % 3) * c.B;
        double* acc_next = c.acc + (size_t)((it + 1) % 3) * c.B;
        double* ex = c.acc + (size_t)(3 + it % 3) * c.B;
        double* ex_next = c.acc + (size_t)(3 + (it + 1) % 3) * c.B;
        for (int b = blockIdx.x * S::TPB + threadIdx.x; b < c.B; b += c.nblocks * S::TPB) {
            acc_next[b] = 0.0;
            ex_next[b] = 0.0;
        }
        // rounds of one vertex per team
        for (int base = 0; base < c.n; base += nt) {
            const int a = base + gteam;
            const int inst = inst_a, out = out_a;
            bool act = false;
            int an = gteam, en = -1;   // the next round's vertex (the first one again after the last round)
            if (rounds && gteam < c.n) {
                if (a + nt < c.n) an = a + nt;
                inst_a = c.vert_inst[an];
                if (tid < 3) en = slot_edge(c, an, tid);
            }
            if (a < c.n) {
                if (!one && done[inst]) bp_copy_vertex<CHI, Mode>(c, a, tid, TB, cur);
                else act = true;
            }
            if (act) bp_front<CHI, Mode, TB>(c, a, tid, team, cur, sm, base == 0 && have_pre, pre, out);
            if (rounds && gteam < c.n && tid < 3) out_a = slot_out(c, an, en);
            if (pend) {
                pend = false;
                const int r = decide(it - 1, dprev);
                if (r < 0) return false;
                if (r > 0) {
                    stop = true;
                    break;
                }
            }
            if (act)
                bp_back<CHI, Mode, TB>(c, tid, team, cur, one ? ex1 : exnow[inst] != 0, sm, one ? nullptr : acc + inst);
        }
        if (stop) break;
        cur ^= 1;
        // one instance: the first warp sums the teams' distances between the block's
        // barrier and its arrival at the grid barrier
        if (!grid_sync_pre(gb, c.spin_limit, [&]() {
                if (!one) return;
                typename Mode::TS v = 0;
                for (int q = threadIdx.x; q < 3 * tpb_teams; q += 32) v += all[q / 3].dsum[q % 3];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (threadIdx.x == 0) atomicAdd(acc, (double)v);
            }))
            return false;
        if (one) dprev = __ldcg(acc);
        if (tid < 3) sm.dsum[tid] = 0;   // read by the first warp before the barrier
        // the next sweep's incoming messages of this team's first vertex are loaded now
        have_pre = false;
        if (gteam < c.n && sm.cached == gteam && tid < 3 * CHI * CHI) {
            const int in = sm.in_idx[tid / (CHI * CHI)];
            if (in >= 0) pre = ldcg((const CT_*)c.msg[cur] + (size_t)in * CHI * CHI + tid % (CHI * CHI));
            have_pre = true;
        }
        ++it;
        if (one) {
            if (AHEAD && it < c.max_iter) {
                pend = true;
                continue;
            }
            const int r = decide(it - 1, dprev);
            if (r < 0) return false;
            if (r > 0) break;
            continue;
        }
        // stopping rule of App. B, per instance, evaluated identically by every block;
        // the raw distance sums are kept and divided by |E| at the end
        const bool last = it >= c.max_iter;
        int open_local = 0, need_local = 0;
        for (int b = threadIdx.x; b < c.B; b += S::TPB) {
            if (done[b]) continue;
            const double dsum = __ldcg(acc + b);
            bool fin;
            if (c.inst_m[b] == 0 || !(dsum == dsum)) {
                fin = true;
            } else if (exnow[b]) {
                fin = last || dsum < thr[b];
            } else if (!last && dsum >= thr_hi[b]) {
                fin = false;   // the exact distance is at least the bound
            } else {
                need[b] = 1;
                need_local = 1;
                continue;
            }
            if (blockIdx.x == 0) {
                c.inst_dist[b] = dsum;
                c.inst_iters[b] = it;
                if (fin) c.inst_done[b] = 1;
            }
            if (fin) done[b] = 1;
            else open_local = 1;
            // the next sweep is exact inline when it is the last or when this
            // sweep came within a factor 3 of the threshold
            exnow[b] = (it + 1 >= c.max_iter) || (float)dsum < thr3[b];
        }
        // one block barrier for both flags (a word per sweep parity, reset one sweep ahead)
        if (need_local | open_local) atomicOr(&sflag[it & 1], need_local | (open_local << 1));
        __syncthreads();
        const int fl = sflag[it & 1];
        if (threadIdx.x == 0) sflag[(it + 1) & 1] = 0;
        if (fl & 1) {
            if (blockIdx.x == 0 && threadIdx.x == 0) ++c.ctl->exact_passes;
            bp_exact_pass<CHI, Mode, S::TPB, TB>(c, cur, need, sm, bsum + 32, ex);
            if (!grid_sync(gb, c.spin_limit)) return false;
            for (int b = threadIdx.x; b < c.B; b += S::TPB) {
                if (!need[b]) continue;
                need[b] = 0;
                const double dsum = __ldcg(ex + b);
                const bool fin = last || dsum < thr[b] || !(dsum == dsum);
                if (blockIdx.x == 0) {
                    c.inst_dist[b] = dsum;
                    c.inst_iters[b] = it;
                    if (fin) c.inst_done[b] = 1;
                }
                if (fin) done[b] = 1;
                else open_local = 1;
                exnow[b] = 1;
            }
            if (!__syncthreads_or(open_local)) break;
        } else if (!(fl & 2)) {
            break;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int mi = 0, ncv = 0;
        double md = 0.0;
        for (int b = 0; b < c.B; ++b) {
            const int mb = c.inst_m[b];
            c.inst_dist[b] = mb > 0 ? c.inst_dist[b] / (double)mb : 0.0;
            mi = c.inst_iters[b] > mi ? c.inst_iters[b] : mi;
            md = c.inst_dist[b] > md ? c.inst_dist[b] : md;
            if (!(c.inst_dist[b] < c.tol) && c.inst_m[b] > 0) ++ncv;
        }
        c.ctl->last_iters = mi;
        c.ctl->last_dist = md;
        c.ctl->not_conv = ncv;
        c.ctl->sweeps_total += mi;
        c.ctl->bp_calls += 1;
        c.ctl->nc_calls += (ncv > 0) ? 1 : 0;
        c.ctl->cur = cur;
    }
    return true;
}

template <int CHI, class Mode, unsigned PH, int V>
__device__ __forceinline__ void anneal_body(const Ctx& c) {
    using S = Shape<CHI, V>;
    extern __shared__ __align__(16) unsigned char smem[];
    GridBarrier gb = grid_barrier_init(c.bar ? c.bar : &c.ctl->bar_count, &c.ctl->err, (unsigned)c.bar_expect);
    const int nteams_total_g = c.nblocks * (S::TPB / S::TG);
    int cur = *(volatile int*)&c.ctl->cur;
    const int kb = c.kdev ? *(volatile int*)c.kdev : c.k0, ke = c.kdev ? kb : c.k1;
    for (int k = kb; k <= ke; ++k) {
        double tZ, tX;
        if (c.Ksched > 0) {
            const double tau = (double)k / (double)c.Ksched;
            tZ = c.dt * tau;
            tX = c.dt * (1.0 - tau);
        } else {
            tZ = c.tZ1;
            tX = c.tX1;
        }
        double sX, cX;
        sincos(tX, &sX, &cX);
        if constexpr ((PH & PH_GATES) != 0u) {
            const double tXp = c.Ksched > 0 ? 0.0 : c.tXpre1;
            const bool pre = tXp != 0.0;
            double sXp = 0.0, cXp = 1.0, sXi = sX, cXi = cX;
            if (pre) {
                sincos(tXp, &sXp, &cXp);
                sincos(tX + tXp, &sXi, &cXi);   // vertices without gates: both mixing gates at once
            }
            const int team = threadIdx.x / S::TG, tid = threadIdx.x % S::TG;
            GateSm<CHI, Mode>& sm = reinterpret_cast<GateSm<CHI, Mode>*>(smem)[team];
            const int gteam = team * c.nblocks + blockIdx.x;
            constexpr int PB = GateSm<CHI, Mode>::PB;
            int seq = 0;   // gates this team has run in the layer
            gate_phases<CHI, Mode>(c, 0, gteam, nteams_total_g, tid, sm, tZ);
            GateMeta next = {};
            if (c.ncol > 0 && c.colour_off[0] + gteam < c.colour_off[1]) next = c.gates[c.colour_off[0] + gteam];
            for (int col = 0; col < c.ncol; ++col) {
                const int beg = c.colour_off[col], end = c.colour_off[col + 1];
                for (int idx = beg + gteam; idx < end; idx += nteams_total_g, ++seq) {
                    const GateMeta gm = next;
                    if (idx + nteams_total_g < end) next = c.gates[idx + nteams_total_g];
                    if (seq % PB == 0 && seq > 0) gate_phases<CHI, Mode>(c, seq, gteam, nteams_total_g, tid, sm, tZ);
                    gate_edge<CHI, Mode>(c, gm, sm.phases + 4 * (seq % PB), tid, team, sm, cX, sX, pre, cXp, sXp);
                }
                if (col == c.ncol - 1)
                    for (int q = gteam; q < c.n_iso; q += nteams_total_g)
                        mixing_vertex<CHI, Mode>(c, c.iso[q], tid, S::TG, cXi, sXi);
                // the next colour's first gate is known before the barrier
                else if (end + gteam < c.colour_off[col + 2])
                    next = c.gates[end + gteam];
                if (!grid_sync(gb, c.spin_limit)) return;
            }
            if (c.ncol == 0) {
                for (int q = gteam; q < c.n_iso; q += nteams_total_g)
                    mixing_vertex<CHI, Mode>(c, c.iso[q], tid, S::TG, cXi, sXi);
                if (!grid_sync(gb, c.spin_limit)) return;
            }
        }
        // regauge policy (Sec. II C): BP and gauge finding only when R exceeds the threshold;
        // every block reads the same value, so the whole grid takes the same branch
        const bool skip_regauge = c.rgate && !(__ldcg(c.rgate) > c.rthr_sum);
        if constexpr ((PH & PH_BP) != 0u) {
            if (skip_regauge) continue;
            {
                static_assert(S::TV == 32, "one warp per BP-init team");
                const int team = threadIdx.x / S::TV, tid = threadIdx.x % S::TV;
                const int gteam = team * c.nblocks + blockIdx.x, nt = c.nblocks * S::NIT;
                double* wsm = reinterpret_cast<double*>(smem) + team * (6 * CHI + 4);
                cd* tsm = reinterpret_cast<cd*>(reinterpret_cast<double*>(smem) + S::NIT * (6 * CHI + 4)) +
                          team * (2 * CHI * CHI * CHI + 3 * CHI * CHI);
                if (team < S::NIT)
                    for (int a = gteam; a < c.n; a += nt)
                        bp_init_vertex<CHI, Mode>(c, a, tid, cur, (c.phases & PH_WARM) != 0, wsm, tsm);
                const int g = blockIdx.x * S::TPB + threadIdx.x;
                for (int b = g; b < c.B; b += c.nblocks * S::TPB) {
                    c.inst_done[b] = 0;   // host-visible copy
                    c.inst_iters[b] = 0;
                    c.inst_dist[b] = 0.0;
                    for (int q = 0; q < 6; ++q) c.acc[q * c.B + b] = 0.0;
                }
                if (!grid_sync(gb, c.spin_limit)) return;
            }
            // FP64 at CHI = 4 while a block's vertices all have a team of four warps: one warp per
            // sub-partition halves a sweep's FP64 time where a block has one vertex (10.4 -> 5.6 us) and
            // evens the sub-partitions out for an odd number; beyond that the teams of two keep every
            // vertex resident
            constexpr int WIDE = SmemSize<CHI, Mode, PH, V>::WIDE_TB;
            bool ok;
            if (WIDE != S::TB && c.n <= c.nsm * (S::TPB / WIDE)) ok = bp_sweeps<CHI, Mode, PH, V, WIDE>(c, gb, cur, smem);
            else ok = bp_sweeps<CHI, Mode, PH, V, S::TB>(c, gb, cur, smem);
            if (!ok) return;
        }
        if constexpr ((PH & PH_REGAUGE) != 0u) {
            if (c.rgate && blockIdx.x == 0 && threadIdx.x == 0) {
                if (skip_regauge) ++c.ctl->reg_skipped;
                else ++c.ctl->regauged;
            }
            if (skip_regauge) continue;
            {
                using SZ = SmemSize<CHI, Mode, PH, V>;
                auto edges = [&](auto lanes, int teams) {
                    constexpr int TEAM = decltype(lanes)::value;
                    const int team = threadIdx.x / TEAM, tid = threadIdx.x % TEAM;
                    if (team >= teams) return;
                    RGSm<CHI>& sm = reinterpret_cast<RGSm<CHI>*>(smem)[team];
                    for (int e = team * c.nblocks + blockIdx.x; e < c.m; e += c.nblocks * teams)
                        regauge_edge<CHI, Mode, TEAM>(c, e, tid, team, cur, sm);
                };
                if (c.m <= c.nsm * (512 / S::TR)) edges(std::integral_constant<int, S::TR>{}, SZ::rg_wide);
                else edges(std::integral_constant<int, S::TR / 2>{}, SZ::rg_teams);
                if (!grid_sync(gb, c.spin_limit)) return;
            }
            {
                using CT = C<typename Mode::TS>;
                const int team = threadIdx.x / S::TRV, tid = threadIdx.x % S::TRV;
                CT* buf = reinterpret_cast<CT*>(smem) + (size_t)team * (4 * CHI * CHI * CHI + 3 * CHI * CHI);
                const int gteam = team * c.nblocks + blockIdx.x, nt = c.nblocks * (S::TPB / S::TRV);
                for (int a = gteam; a < c.n; a += nt) {
                    regauge_vertex<CHI, Mode, S::TRV>(c, a, tid, team, buf);
                    team_bar<S::TRV>(team);
                }
                if (!grid_sync(gb, c.spin_limit)) return;
            }
        }
        // every block read *kdev at entry, before the barriers above
        if constexpr ((PH & PH_REGAUGE) != 0u)
            if (c.kdev && blockIdx.x == 0 && threadIdx.x == 0) *c.kdev = k + 1;
    }
}

// The three phase kernels (one cooperative launch each).
template <int CHI, class Mode, int V>
__global__ void __launch_bounds__(Shape<CHI, V>::TPB, 1) gates_kernel(Ctx c) { anneal_body<CHI, Mode, PH_GATES, V>(c); }
template <int CHI, class Mode, int V>
__global__ void __launch_bounds__(Shape<CHI, V>::TPB, 1) bp_kernel(Ctx c) { anneal_body<CHI, Mode, PH_BP, V>(c); }
template <int CHI, class Mode, int V>
__global__ void __launch_bounds__(Shape<CHI, V>::TPB, 1) regauge_kernel(Ctx c) {
    anneal_body<CHI, Mode, PH_REGAUGE, V>(c);
}

}  // namespace gtqa
