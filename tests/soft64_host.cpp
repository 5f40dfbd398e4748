// vamp_soft64.cuh compiled for the host: its functions over arrays, a call
// a function, for test_soft64.py.
#include "../paper_1811_09711_gb300/csrc/vamp_soft64.cuh"

using namespace vamp;

namespace {
// value = m 2^e
void put(Sf a, uint64_t* m, int* e, int i)
{
    m[i] = a.m;
    e[i] = a.e;
}
}  // namespace

extern "C" {

void t_exp2(int n, const double* x, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) put(sf_exp2(x[i]), m, e, i);
}

// log2 x as ±m 2^e: the sign in s
void t_log2(int n, const double* x, uint64_t* m, int* e, int* s)
{
    for (int i = 0; i < n; ++i) {
        bool neg;
        put(sf_log2(sf_from_double(x[i]), neg), m, e, i);
        s[i] = neg ? -1 : 1;
    }
}

void t_pow(int n, const double* x, const double* y, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) put(sf_pow(sf_from_double(x[i]), y[i]), m, e, i);
}

}
