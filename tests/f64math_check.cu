// Host driver for csrc/f64math.cuh (compiled by nvcc for the host only;
// tests/test_f64math_host.py checks the answers): one float64 (hex bits) per
// line on stdin -> sqrt, 1 / sqrt, 1 / x, log(1 + x), log x (hex bits).
#include <stdio.h>

#include "f64math.cuh"

int main()
{
    unsigned long long b;
    while (scanf("%llx", &b) == 1) {
        const double x = hts::double_of(b);
        double t, rs;
        hts::sqrt_rsqrt(x, t, rs);
        printf("%llx %llx %llx %llx %llx\n", hts::bits_of(t), hts::bits_of(rs), hts::bits_of(hts::reciprocal(x)),
               hts::bits_of(hts::log1p_pos(x)), hts::bits_of(hts::log_pos(x)));
    }
    return 0;
}
