// Host build of the integer double arithmetic for test_soft64.py.
#include "soft64.cuh"

extern "C" {
double s64h_mul(double a, double b) { return ck::s64_mul(a, b); }
int s64h_in_range(double a) { return ck::s64_ok(ck::s64_range(a)); }
float s64h_to_float(double a, int *ok) {
    bool k = true;
    const float f = ck::s64_to_float(a, k);
    *ok = k;
    return f;
}
double s64h_from_float(float a) { return ck::s64_from_float(a); }
}
