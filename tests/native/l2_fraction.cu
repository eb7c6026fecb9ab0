// Host-side check of l2_keep_fraction (skf_internal.cuh): the fraction of a
// createpolicy.fractional lies in (0, 1] for every operator size.  Prints the
// number of checked sizes and of values outside; exits 1 if there is one.
#include "../../paper_2208_11447_gb300/csrc/skf_internal.cuh"

#include <cstdio>

int main() {
    long checked = 0, bad = 0;
    for (double b = 1.0; b < 1e13; b *= 1.001, ++checked) {
        const float f = skf::l2_keep_fraction(b);
        if (!(f > 0.f && f <= 1.f)) ++bad;
    }
    printf("checked %ld outside %ld\n", checked, bad);
    return bad != 0;
}
