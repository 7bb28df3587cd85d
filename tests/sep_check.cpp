// The separable factors of csrc/sep_factors.h as a shared library for tests/test_sep_factors_cpu.py.
#include "sep_factors.h"

extern "C" int sep_check(const double *E, int nv, int nc, int max_terms, int *ldu, float *tab, float *scale, long cap)
{
    const gw::SepFactors f = gw::sep_factors(E, nv, nc, 16, max_terms);
    *ldu = f.ldu;
    if ((long)f.tab.size() > cap)
        return -1;
    for (size_t i = 0; i < f.tab.size(); ++i)
        tab[i] = f.tab[i];
    for (size_t i = 0; i < f.scale.size(); ++i)
        scale[i] = f.scale[i];
    return f.T;
}
