// The sines of the central column pass (eighth_sine, fftconv.cuh) on the CPU: for
// every transform length and bin, from table entries rounded as k_phase rounds
// them, the largest relative error in units of the precision's rounding.
#include "../paper_2001_02765_gb300/csrc/fftconv.cuh"

#include <cmath>
#include <cstdio>

template <typename T>
static double worst(int py, double h)
{
    using C = cplx_t<T>;
    auto entry = [&](int k) {
        const double t = 2.0 * M_PI * k / py;
        return cmake<C>((T)(cos(t) / (2.0 * h)), (T)(sin(t) / (2.0 * h)));
    };
    const int step = py / 8;
    double w = 0.0;
    for (int jt = 0; jt < step; ++jt)
        for (int q = 0; q < 8; ++q) {
            const long double ref = sinl(2.0L * M_PIl * (jt + q * step) / py) / (2.0L * (long double)h);
            const long double d = (long double)sgk::eighth_sine(entry(jt), entry(step - jt), q) - ref;
            if ((jt + q * step) % (py / 2) == 0) {  // sin 0 and sin pi
                if (fabsl(d) > 1e-15 / h) return 1e9;
            } else {
                w = fmax(w, (double)(fabsl(d / ref) / (sizeof(T) == 4 ? 0x1p-24L : 0x1p-53L)));
            }
        }
    return w;
}

int main()
{
    for (int L = SG_MIN_PAD; L <= SG_MAX_PAD; L = sg_next_length(L))
        printf("%d %.3f %.3f\n", L, worst<float>(L, 0.0137), worst<double>(L, 0.0137));
    return 0;
}
