// Test helper (not part of the library): what the relaxation rates s_q and
// sigma_e, which vanish with the viscosity, do to a node in FP32 and in FP64,
// compiled for the CPU, for tests/test_node_rates.py.
#include <cstddef>

#include "../paper_1809_08683_gb300/csrc/lbm_node.cuh"

template <typename R>
static lbm::Params<R> params(double mu0, double mu_j, double nu_e) {
    lbm::Params<R> P{};
    P.rho0 = P.T0 = P.inv_T0 = P.Cv = P.inv_Cv = P.Rg = P.hh = R(1);
    P.mu0 = R(mu0);
    P.mu_j = R(mu_j);
    P.nu_e = R(nu_e);
    P.eos = lbm::EOS_IDEAL;
    return P;
}

struct TakeIncrement {  // of the population g[0]
    double* out;
    const void* g0;
    template <typename R>
    void operator()(R&, R, R& g, R dg) const {
        if (&g == g0) *out = (double)dg;
    }
};

// Increment of g_0 of a node at rest whose only moment is n_1 = 36: a
// multiple of sigma_e alone.
template <typename R>
static double sigma_e(double mu0, double mu_j) {
    const lbm::Params<R> P = params<R>(mu0, mu_j, 1.0);
    R f[9] = {}, g[9] = {R(-4), R(-1), R(-1), R(-1), R(-1), R(2), R(2), R(2), R(2)}, rd, jx, jy, sg;
    lbm::Mac<R> m;
    lbm::node_sums(f, g, rd, jx, jy, sg);
    lbm::macros(P, rd, jx, jy, sg, m);
    double out = 0.0;
    lbm::collide(P, m, f, g, R(0), R(0), R(0), R(0), TakeIncrement{&out, g});
    return out;
}

// Row 1 of (I - S/2) d for d = e_4, u = (1, 0) and s_e small: a multiple of s_q.
template <typename R>
static double s_q(double mu0) {
    const lbm::Params<R> P = params<R>(mu0, 1.0, 1e6);
    lbm::Rates<R> r;
    lbm::rates(P, R(1), R(1), r);
    lbm::Dev<R> d{};
    d.d4 = R(1);
    lbm::Gv<R> G;
    lbm::apply_IS2(P, r, R(1), R(0), d, G);
    return (double)G.G1;
}

extern "C" void node_rates(double mu0, double mu_j, double* fp32, double* fp64) {
    fp32[0] = sigma_e<float>(mu0, mu_j);
    fp64[0] = sigma_e<double>(mu0, mu_j);
    fp32[1] = s_q<float>(mu0);
    fp64[1] = s_q<double>(mu0);
}
