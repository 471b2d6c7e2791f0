// Plain-path kernel instantiations.  pm selects the precision: 0 FP64 and 1 mixed (complex64
// storage and contractions; FP64 QR/SVD, gauge roots and normalisation), each for degree 4 with
// CHI in {2, 4} and degree 3 with CHI = 16; 2 the complex64 mode (every step in FP32), for
// degree 3 with CHI in {2, 4, 8, 16} and degree 4 with CHI in {2, 4}.
#include "gtqa_launch.h"

namespace gtqa {

namespace {
template <int CHI, int D, typename R, typename RC>
cudaError_t init_t(const PlainArgs& a, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    plain_bp_init_kernel<CHI, D, R, RC><<<a.n, 256, PlainShape<CHI, D, R, RC>::init_smem, st>>>(a);
    return cudaGetLastError();
}
template <int CHI, int D, typename R, typename RC>
cudaError_t bp_t(const PlainBPArgs& a, cudaStream_t st) {
    PlainBPArgs copy = a;
    void* args[] = {&copy};
    return cudaLaunchCooperativeKernel((const void*)plain_bp_kernel<CHI, D, R, RC>, dim3(a.nblocks), dim3(512), args,
                                       PlainShape<CHI, D, R, RC>::bp_smem, st);
}
template <int CHI, int D, typename R, typename RC>
cudaError_t regauge_t(const PlainArgs& a, double eig_cut, double svd_cut, cudaStream_t st) {
    using S = PlainShape<CHI, D, R, R>;
    if (a.m > 0) {
        plain_regauge_edge_kernel<CHI, R, RC><<<a.m, S::CC, sizeof(PlainEdgeSm<CHI, RC>), st>>>(a, eig_cut, svd_cut);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (a.n <= 0) return cudaSuccess;
    plain_regauge_vertex_kernel<CHI, D, R><<<2 * a.n, S::NT, S::vertex_smem, st>>>(a);
    return cudaGetLastError();
}
// the shared-memory limits of the kernels of one shape
template <int CHI, int D, typename R, typename RC>
cudaError_t prepare_t() {
    using S = PlainShape<CHI, D, R, RC>;
    cudaError_t e = raise_smem_limit(plain_bp_init_kernel<CHI, D, R, RC>, S::init_smem);
    if (e == cudaSuccess) e = raise_smem_limit(plain_bp_kernel<CHI, D, R, RC>, S::bp_smem);
    if (e == cudaSuccess) e = raise_smem_limit(plain_regauge_edge_kernel<CHI, R, RC>, sizeof(PlainEdgeSm<CHI, RC>));
    if (e == cudaSuccess) e = raise_smem_limit(plain_regauge_vertex_kernel<CHI, D, R>, PlainShape<CHI, D, R, R>::vertex_smem);
    return e;
}
template <int CHI, int D, typename R>
cudaError_t marg_t(const void* G, const double* lam, const int4* vs, int n, cd* rho, int8_t* sign, int* flag,
                   cudaStream_t st) {
    const int wpb = 4;
    plain_marginals_kernel<CHI, D, R><<<(n + wpb - 1) / wpb, 32 * wpb, 0, st>>>((const C<R>*)G, lam, vs, n, rho, sign,
                                                                                flag);
    return cudaGetLastError();
}
template <int CHI, int D, typename R>
cudaError_t resid_t(const void* G, const double* lam, const int4* vs, int n, double* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    plain_residual_kernel<CHI, D, R><<<n * D, PlainShape<CHI, D, R>::CC / 2, 0, st>>>((const C<R>*)G, lam, vs, out);
    return cudaGetLastError();
}
template <int CHI, int D, typename R>
cudaError_t sample_t(void* G, const double* lam, const int4* vs, int a, double u, int step, int8_t* x, double* p,
                     cudaStream_t st) {
    plain_sample_kernel<CHI, D, R><<<1, 32, 0, st>>>((C<R>*)G, lam, vs, a, u, step, x, p);
    return cudaGetLastError();
}
}  // namespace

// CALL(CHI, D, R, RC) for every built shape: R the storage and contraction type, RC the type
// of the FP64 steps (normalisation, trace norms, the regauge's eigen and SVD)
#define GTQA_PLAIN_DISPATCH(CALL)                                              \
    if (pm == 0) {                                                             \
        if (D == 4 && CHI == 2) return CALL(2, 4, double, double);             \
        if (D == 4 && CHI == 4) return CALL(4, 4, double, double);             \
        if (D == 3 && CHI == 16) return CALL(16, 3, double, double);           \
    } else if (pm == 1) {                                                      \
        if (D == 4 && CHI == 2) return CALL(2, 4, float, double);              \
        if (D == 4 && CHI == 4) return CALL(4, 4, float, double);              \
        if (D == 3 && CHI == 16) return CALL(16, 3, float, double);            \
    } else {                                                                   \
        if (D == 3 && CHI == 2) return CALL(2, 3, float, float);               \
        if (D == 3 && CHI == 4) return CALL(4, 3, float, float);               \
        if (D == 3 && CHI == 8) return CALL(8, 3, float, float);               \
        if (D == 3 && CHI == 16) return CALL(16, 3, float, float);             \
        if (D == 4 && CHI == 2) return CALL(2, 4, float, float);               \
        if (D == 4 && CHI == 4) return CALL(4, 4, float, float);               \
    }                                                                          \
    return cudaErrorInvalidValue;

bool plain_supported(int CHI, int D, int pm) {
    if (pm != 2) return (D == 4 && (CHI == 2 || CHI == 4)) || (D == 3 && CHI == 16);
    return (D == 3 && (CHI == 2 || CHI == 4 || CHI == 8 || CHI == 16)) || (D == 4 && (CHI == 2 || CHI == 4));
}

size_t plain_scratch_entries(int CHI, int D, int gates) {
    // complex entries: the reflectors of the largest launch of CHI = 16 gates
    return D == 3 && CHI == 16 ? (size_t)gates * 4 * 16 * 256 : 0;
}

cudaError_t plain_prepare(int CHI, int D, int pm) {
#define C_(c, d, r, rc) prepare_t<c, d, r, rc>()
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_bp_init_launch(int CHI, int D, int pm, const PlainArgs& a, cudaStream_t st) {
#define C_(c, d, r, rc) init_t<c, d, r, rc>(a, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_bp_launch(int CHI, int D, int pm, const PlainBPArgs& a, cudaStream_t st) {
#define C_(c, d, r, rc) bp_t<c, d, r, rc>(a, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_regauge_launch(int CHI, int D, int pm, const PlainArgs& a, double eig_cut, double svd_cut,
                                 cudaStream_t st) {
#define C_(c, d, r, rc) regauge_t<c, d, r, rc>(a, eig_cut, svd_cut, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_marginals_launch(int CHI, int D, int pm, const void* G, const double* lam, const int4* vs, int n,
                                   cd* rho, int8_t* sign, int* flag, cudaStream_t st) {
#define C_(c, d, r, rc) marg_t<c, d, r>(G, lam, vs, n, rho, sign, flag, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_residual_launch(int CHI, int D, int pm, const void* G, const double* lam, const int4* vs, int n,
                                  double* out, cudaStream_t st) {
#define C_(c, d, r, rc) resid_t<c, d, r>(G, lam, vs, n, out, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_sample_launch(int CHI, int D, int pm, void* G, const double* lam, const int4* vs, int a, double u,
                                int step, int8_t* x, double* p, cudaStream_t st) {
#define C_(c, d, r, rc) sample_t<c, d, r>(G, lam, vs, a, u, step, x, p, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_general_gates_launch(int CHI, int D, int pm, const GenArgs& a, cudaStream_t st) {
    if (pm == 0) {
        if (D == 4 && CHI == 2) return general_gates_launch_t<2, 4, ModeFP64>(a, st);
        if (D == 4 && CHI == 4) return general_gates_launch_t<4, 4, ModeFP64>(a, st);
    } else if (pm == 1) {
        if (D == 4 && CHI == 2) return general_gates_launch_t<2, 4, ModeMixed>(a, st);
        if (D == 4 && CHI == 4) return general_gates_launch_t<4, 4, ModeMixed>(a, st);
    } else {
        if (D == 3 && CHI == 2) return general_gates_launch_t<2, 3, ModeC64>(a, st);
        if (D == 3 && CHI == 4) return general_gates_launch_t<4, 3, ModeC64>(a, st);
        if (D == 3 && CHI == 8) return general_gates_launch_t<8, 3, ModeC64>(a, st);
        if (D == 4 && CHI == 2) return general_gates_launch_t<2, 4, ModeC64>(a, st);
        if (D == 4 && CHI == 4) return general_gates_launch_t<4, 4, ModeC64>(a, st);
    }
    return cudaErrorInvalidValue;   // CHI = 16: the whole-side core (64 x 64) exceeds one block's Jacobi
}
cudaError_t plain_single_gates_launch(int CHI, int D, int pm, void* G, const int* v, const cd* W, int count,
                                      cudaStream_t st) {
    if (pm == 0) {
        if (D == 4 && CHI == 2) return single_gates_launch_t<2, 4, ModeFP64>(G, v, W, count, st);
        if (D == 4 && CHI == 4) return single_gates_launch_t<4, 4, ModeFP64>(G, v, W, count, st);
        if (D == 3 && CHI == 16) return single_gates_launch_t<16, 3, ModeFP64>(G, v, W, count, st);
    } else if (pm == 1) {
        if (D == 4 && CHI == 2) return single_gates_launch_t<2, 4, ModeMixed>(G, v, W, count, st);
        if (D == 4 && CHI == 4) return single_gates_launch_t<4, 4, ModeMixed>(G, v, W, count, st);
        if (D == 3 && CHI == 16) return single_gates_launch_t<16, 3, ModeMixed>(G, v, W, count, st);
    } else {
        if (D == 3 && CHI == 2) return single_gates_launch_t<2, 3, ModeC64>(G, v, W, count, st);
        if (D == 3 && CHI == 4) return single_gates_launch_t<4, 3, ModeC64>(G, v, W, count, st);
        if (D == 3 && CHI == 8) return single_gates_launch_t<8, 3, ModeC64>(G, v, W, count, st);
        if (D == 3 && CHI == 16) return single_gates_launch_t<16, 3, ModeC64>(G, v, W, count, st);
        if (D == 4 && CHI == 2) return single_gates_launch_t<2, 4, ModeC64>(G, v, W, count, st);
        if (D == 4 && CHI == 4) return single_gates_launch_t<4, 4, ModeC64>(G, v, W, count, st);
    }
    return cudaErrorInvalidValue;
}

namespace {
template <int CHI, int D, typename TS, typename R>
cudaError_t ising_t(const PlainGateArgs* a, cudaStream_t st) {
    if constexpr (CHI == 16) {
        constexpr size_t smem = sizeof(Gate16Sm<R>);
        if (!a) return raise_smem_limit(ising16_gate_kernel<TS, R>, smem);
        ising16_gate_kernel<TS, R><<<a->count, 512, smem, st>>>(*a);
    } else {
        constexpr size_t smem = sizeof(PlainGateSm<CHI, D, TS, R>);
        if (!a) return raise_smem_limit(plain_ising_kernel<CHI, D, TS, R>, smem);
        plain_ising_kernel<CHI, D, TS, R><<<a->count, PlainGateShape<CHI, D>::TEAM, smem, st>>>(*a);
    }
    return cudaGetLastError();
}
template <int CHI, int D, typename TS>
cudaError_t mixing_t(void* G, const int* v, int count, double c, double s, cudaStream_t st) {
    plain_mixing_kernel<CHI, D, TS><<<count, 64, 0, st>>>(G, v, c, s);
    return cudaGetLastError();
}
}  // namespace

// a = nullptr: only raises the kernel's shared-memory limit (once per state, at creation)
cudaError_t plain_ising_launch(int CHI, int D, int pm, const PlainGateArgs* a, cudaStream_t st) {
    if (a && a->count <= 0) return cudaSuccess;
#define C_(c, d, r, rc) ising_t<c, d, r, rc>(a, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}
cudaError_t plain_mixing_launch(int CHI, int D, int pm, void* G, const int* v, int count, double cs, double sn,
                                cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
#define C_(c, d, r, rc) mixing_t<c, d, r>(G, v, count, cs, sn, st)
    GTQA_PLAIN_DISPATCH(C_)
#undef C_
}

}  // namespace gtqa
