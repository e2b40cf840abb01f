// Host driver of the divide and conquer eigensolver in evc_dc.cuh: the phases
// of its device driver, each run by one thread.
#include <cmath>
#include <vector>

#include "evc_dc.cuh"

using namespace evc;

extern "C" void dc_eig(int k, const double* diag, const double* off, double* theta, double* first)
{
    std::vector<double> buf(dc_smem(k) / sizeof(double) + 2), e(off, off + k - 1);
    DcWork w = dc_carve(buf.data(), k);
    int ex = -100000;
    for (int t = 0; t < k; ++t) {
        const double m = std::fmax(std::fabs(diag[t]), t + 1 < k ? std::fabs(e[t]) : 0.0);
        if (m > 0.0) ex = std::max(ex, std::ilogb(m) + 1);
    }
    if (ex == -100000) ex = 0;
    for (int t = 0; t < k; ++t) {
        w.d[t] = std::scalbn(diag[t], -ex);
        if (t + 1 < k) e[t] = std::scalbn(e[t], -ex);
        w.f[t] = w.l[t] = 1.0;
    }
    for (int t = 0; t < k; t += 2) {
        const double a = t > 0 ? std::fabs(e[t - 1]) : 0.0, b = t + 2 < k ? std::fabs(e[t + 1]) : 0.0;
        if (t + 1 < k) dc_pair(w.d[t] - a, e[t], w.d[t + 1] - b, w.d + t, w.f + t, w.l + t);
        else w.d[t] -= a;
    }
    const DcLanes ln{0, 1, 1};
    for (int half = 2; half < k; half *= 2) {
        DcLevel L{w, e.data(), k, half, 1};
        L.sort(0, 1);
        L.flag(0, 1);
        L.keep(0, 1);
        bool any = false;
        for (int g = 0; g < k; ++g) any = any || L.close(g);
        if (any) {
            for (int g = 0; g < k; ++g)
                if (L.beg(g) == g) L.deflate_close(g);
            L.keep(0, 1);
        }
        for (int g = 0; g < k; ++g) L.roots<1>(g, ln);
        for (int g = 0; g < k; ++g) L.loewner<1>(g, ln);
        for (int g = 0; g < k; ++g) L.vectors<1>(g, ln);
        L.order(0, 1);
        L.swap();
        w = L.w;
    }
    for (int t = 0; t < k; ++t) {
        theta[t] = std::scalbn(w.d[t], ex);
        first[t] = w.f[t];
    }
}
