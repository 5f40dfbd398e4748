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

void t_rcp(int n, const double* x, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) put(sf_rcp(sf_from_double(x[i])), m, e, i);
}

void t_any_rcp(int n, const double* x, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) put(sf_rcp(sf_from_any(x[i])), m, e, i);
}

void t_powm08(int n, const double* x, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) put(sf_powm08(x[i]), m, e, i);
}

// x y x y x y x y, normalised at the end
void t_products(int n, const double* x, const double* y, uint64_t* m, int* e)
{
    for (int i = 0; i < n; ++i) {
        Sf p{1ull << 63, -63};
        for (int q = 0; q < 8; ++q) p = sf_mul(p, sf_from_double(q & 1 ? y[i] : x[i]));
        put(sf_norm(p), m, e, i);
    }
}

// results that are doubles
void t_tan(int n, const double* x, double* r)
{
    for (int i = 0; i < n; ++i) r[i] = sf_tan(x[i]);
}

void t_div(int n, const double* x, const double* y, double* r)
{
    for (int i = 0; i < n; ++i) r[i] = sf_div(x[i], y[i]);
}

}
