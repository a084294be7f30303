// Host driver for csrc/polar.cuh (compiled by nvcc for the host only;
// tests/test_polar_host.py checks the answers): per line on stdin x, y, lo, hi
// (float64 hex bits) and the split rule -> whether the pairs decide the angle
// and the radius, and their quantised values.
#include <stdio.h>

#include "polar.cuh"

int main()
{
    unsigned long long b[4];
    int area;
    while (scanf("%llx %llx %llx %llx %d", b, b + 1, b + 2, b + 3, &area) == 5) {
        const double x = hts::double_of(b[0]), y = hts::double_of(b[1]);
        const hts::RadialBounds r = hts::radial_bounds(hts::double_of(b[2]), hts::double_of(b[3]));
        volatile double xx = x * x, yy = y * y;  // each operation rounded on its own
        uint64_t qa = 0, qr = 0;
        const int a = hts::quantise_angle(x, y, 29, qa), c = hts::quantise_radius(xx + yy, area != 0, r, 29, qr);
        printf("%d %llu %d %llu\n", a, (unsigned long long)qa, c, (unsigned long long)qr);
    }
    return 0;
}
