// Host build of the comparisons and conversions of the integer double arithmetic for test_soft64_compare.py.
#include "soft64.cuh"

extern "C" {
int s64c_le_pos(double a, double b) { return ck::s64_le_pos(a, b); }
int s64c_gt_pos(double a, double b) { return ck::s64_gt_pos(a, b); }
int s64c_positive(double a) { return ck::s64_positive(a); }
int s64c_not_positive(double a) { return ck::s64_not_positive(a); }
int s64c_not_negative(double a) { return ck::s64_not_negative(a); }
int s64c_isnan(double a) { return ck::s64_isnan(a); }
int s64c_is_zero(double a) { return ck::s64_is_zero(a); }
float s64c_truncate(double a) { return ck::s64_truncate(a); }
}
