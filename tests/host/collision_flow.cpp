// Periodic flows advanced by the library's collision functions in three
// arithmetics: double (what FP64 storage runs), Dual<double> (its value parts
// take the equilibria through the moment cube, in double) and long double.
// Arguments: nx ny nz U amplitude hkind (trt | cum1st) T_ref steps seed.
// Prints the relative L2 errors of f and h against long double in the first and
// the second, then the change of mass and energy per node of the first.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "lbm_device.cuh"

using namespace lbmd;
typedef long double L;

static double value(double x) { return x; }
static double value(Dual<double> x) { return x.v; }
static L value(L x) { return x; }

template <typename R> struct Flow {
    int nx, ny, nz, N;
    bool cum;
    DevParams p;
    std::vector<R> f, h, f2, h2;  // [27][N] deviations
    Flow(int x, int y, int z, bool cumulants, double Tref)
        : nx(x), ny(y), nz(z), N(x * y * z), cum(cumulants), p(), f(27 * N), h(27 * N), f2(27 * N), h2(27 * N) {
        const double nu = 0.02, k = 1e-3, s = 1.0 / (3.0 * k + 0.5);
        p.omega1 = 1.0 / (3.0 * nu + 0.5);
        p.omega_bulk = 1.0;
        p.rho0 = 1.0;
        p.Tref = Tref;
        for (int o = 0; o < 7; ++o) p.sh[o] = cum ? (o == 1 ? s : 1.0) : (o % 2 ? s : 1.0);
        sync_float_params(p);
    }
    void init(const std::vector<double>& v) {  // per node: rho - rho0, rho T - T_ref, u
        for (int n = 0; n < N; ++n) {
            R a[27], b[27];
            feq_dev<R>(a, R(v[5 * n]), R(v[5 * n + 2]), R(v[5 * n + 3]), R(v[5 * n + 4]), p);
            heq_dev<R, 27>(b, R(v[5 * n + 1]), R(v[5 * n + 2]), R(v[5 * n + 3]), R(v[5 * n + 4]), p);
            for (int i = 0; i < 27; ++i) f[i * N + n] = a[i], h[i * N + n] = b[i];
        }
    }
    template <typename Q> void start_from(const Flow<Q>& o) {
        for (int i = 0; i < 27 * N; ++i) f[i] = R(value(o.f[i])), h[i] = R(value(o.h[i]));
    }
    void step() {
        for (int n = 0; n < N; ++n) {
            const int x = n % nx, y = n / nx % ny, z = n / (nx * ny);
            R a[27], b[27], ux, uy, uz, rho;
            for (int i = 0; i < 27; ++i) {
                const int m = (x - EX(i) + nx) % nx + nx * ((y - EY(i) + ny) % ny + ny * ((z - EZ(i) + nz) % nz));
                a[i] = f[i * N + m];
                b[i] = h[i * N + m];
            }
            collide_f<R>(a, p, ux, uy, uz, rho);
            if (cum) collide_h<R, 27, true, false>(b, ux, uy, uz, R(0), p);
            else collide_h<R, 27, false, true>(b, ux, uy, uz, R(0), p);
            for (int i = 0; i < 27; ++i) f2[i * N + n] = a[i], h2[i * N + n] = b[i];
        }
        f.swap(f2);
        h.swap(h2);
    }
};

template <typename R> static double error(const std::vector<R>& v, const std::vector<L>& ref) {
    L d = 0, s = 0;
    for (size_t i = 0; i < v.size(); ++i) {
        d += (value(v[i]) - ref[i]) * (value(v[i]) - ref[i]);
        s += ref[i] * ref[i];
    }
    return s > 0 ? (double)sqrtl(d / s) : (double)sqrtl(d);
}
static L total(const std::vector<double>& v) {
    L t = 0;
    for (double x : v) t += x;
    return t;
}

int main(int argc, char** argv) {
    if (argc != 10) return 2;
    const int nx = atoi(argv[1]), ny = atoi(argv[2]), nz = atoi(argv[3]), steps = atoi(argv[8]);
    const double U = atof(argv[4]), amp = atof(argv[5]), Tref = atof(argv[7]);
    const bool cum = !strcmp(argv[6], "cum1st");
    uint32_t r = (uint32_t)atoi(argv[9]);
    auto random = [&] { return ((r = r * 1664525u + 1013904223u) >> 8) / 16777216.0 - 0.5; };
    Flow<L> a(nx, ny, nz, cum, Tref);
    Flow<double> b(nx, ny, nz, cum, Tref);
    Flow<Dual<double>> c(nx, ny, nz, cum, Tref);
    std::vector<double> v(5 * a.N);
    for (int n = 0; n < a.N; ++n) {
        v[5 * n] = amp * random();
        v[5 * n + 1] = amp * random();
        for (int d = 0; d < 3; ++d) v[5 * n + 2 + d] = U * random();
    }
    c.init(v);
    a.start_from(c);
    b.start_from(c);
    const L m0 = total(b.f), e0 = total(b.h);
    for (int t = 0; t < steps; ++t) {
        a.step();
        b.step();
        c.step();
    }
    printf("%.6e %.6e %.6e %.6e %.6e %.6e\n", error(b.f, a.f), error(b.h, a.h), error(c.f, a.f), error(c.h, a.h),
           (double)((total(b.f) - m0) / a.N), (double)((total(b.h) - e0) / a.N));
    return 0;
}
