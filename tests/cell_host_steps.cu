// cell_host_steps.cu -- host build of the collisions that the FP64 steps and the plain and
// Powell FP32 steps run (ideal_cell.cuh: ideal_collide_f64, powell_collide and ideal_collide_hom
// with the constants from a table, ideal_collide_f32), for CPU tests against the oracle.  Test
// infrastructure only; beside cell_host.cu, whose plain entries are the corrected step's form.
//
// Each entry collides one cell's populations f[k * q + i] in place with the kernels' own inputs
// (omega_k, src0_k = w_0 S_k, src1_k = w_moving S_k) and returns 0, or -1 for a dimension other
// than 2 or 3.  Status bits a cell raises are OR-ed into *flags.
#include "ideal_cell.cuh"

using namespace vlbm;

namespace {

template <int D, int NL, class C, class F> void on_cell(C *f, F collide)
{
    constexpr int Q = AxisSet<D>::Q;
    C c[NL][Q];
    for (int k = 0; k < NL; ++k)
        for (int i = 0; i < Q; ++i) c[k][i] = f[k * Q + i];
    collide(c);
    for (int k = 0; k < NL; ++k)
        for (int i = 0; i < Q; ++i) f[k * Q + i] = c[k][i];
}

template <int D> RelaxTable<double, kMaxLat> table(const double *omega, int nl)
{
    RelaxTable<double, kMaxLat> t{};
    for (int k = 0; k < nl; ++k) t.relax[k] = relax_of<D, double>(omega[k]);
    return t;
}

template <int D>
void f64(double gm1, const double *omega, const double *src0, const double *src1, double *f, unsigned *flags)
{
    const auto t = table<D>(omega, 8);
    on_cell<D, 8>(f, [&](auto &c) { ideal_collide_f64<D, double>(c, gm1, t, src0, src1, flags); });
}

template <int D>
void powell_f64(double gm1, const double *omega, const double *src0, const double *src1, double inv_tau_m, double *f,
                unsigned *flags)
{
    const auto t = table<D>(omega, 9);
    on_cell<D, 9>(f, [&](auto &c) { powell_collide<D, double>(c, gm1, t, src0, src1, inv_tau_m, flags); });
}

template <int D>
void hom_f64(double gm1, const double *omega, const double *src0, const double *src1, double d, const double *uB,
             const double *BB, double *f, unsigned *flags)
{
    const auto t = table<D>(omega, 8);
    const double u[3] = {uB[0], uB[1], uB[2]}, b[3] = {BB[0], BB[1], BB[2]};
    on_cell<D, 8>(f, [&](auto &c) { ideal_collide_hom<D, double>(c, gm1, t, src0, src1, flags, d, u, b); });
}

template <int D, int NL>
void f32(float gm1, const float *omega, const float *src0, const float *src1, float inv_tau_m, float *f, unsigned *flags)
{
    auto relax = [&](int k) { return relax_source<D>(omega[k], src0[k], src1[k]); };
    on_cell<D, NL>(f, [&](auto &c) { ideal_collide_f32<D, NL>(c, gm1, relax, flags, inv_tau_m); });
}

}  // namespace

#define HC_DIM(dim, call2, call3) \
    do {                          \
        if ((dim) == 2) {         \
            call2;                \
        } else if ((dim) == 3) {  \
            call3;                \
        } else {                  \
            return -1;            \
        }                         \
        return 0;                 \
    } while (0)

extern "C" {

int hs_ideal_f64(int dim, double gm1, const double *omega, const double *src0, const double *src1, double *f,
                 unsigned *flags)
{
    HC_DIM(dim, f64<2>(gm1, omega, src0, src1, f, flags), f64<3>(gm1, omega, src0, src1, f, flags));
}

int hs_powell_f64(int dim, double gm1, const double *omega, const double *src0, const double *src1, double inv_tau_m,
                  double *f, unsigned *flags)
{
    HC_DIM(dim, powell_f64<2>(gm1, omega, src0, src1, inv_tau_m, f, flags),
           powell_f64<3>(gm1, omega, src0, src1, inv_tau_m, f, flags));
}

int hs_hom_f64(int dim, double gm1, const double *omega, const double *src0, const double *src1, double d,
               const double *uB, const double *BB, double *f, unsigned *flags)
{
    HC_DIM(dim, hom_f64<2>(gm1, omega, src0, src1, d, uB, BB, f, flags),
           hom_f64<3>(gm1, omega, src0, src1, d, uB, BB, f, flags));
}

int hs_ideal_f32(int dim, float gm1, const float *omega, const float *src0, const float *src1, float *f,
                 unsigned *flags)
{
    HC_DIM(dim, (f32<2, 8>(gm1, omega, src0, src1, 0.f, f, flags)), (f32<3, 8>(gm1, omega, src0, src1, 0.f, f, flags)));
}

int hs_powell_f32(int dim, float gm1, const float *omega, const float *src0, const float *src1, float inv_tau_m,
                  float *f, unsigned *flags)
{
    HC_DIM(dim, (f32<2, 9>(gm1, omega, src0, src1, inv_tau_m, f, flags)),
           (f32<3, 9>(gm1, omega, src0, src1, inv_tau_m, f, flags)));
}

}  // extern "C"
