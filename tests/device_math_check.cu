// Device driver for csrc/polar.cuh and csrc/f64math.cuh (tests/test_gpu_device_math.py
// checks the answers).  "polar": per line on stdin x, y, lo, hi (float64 hex bits)
// and the split rule -> as polar_check.cu; "math": per line one float64 -> as
// f64math_check.cu.
#include <stdio.h>
#include <string.h>

#include <vector>

#include "f64math.cuh"
#include "polar.cuh"

struct Row {
    unsigned long long b[5];
};

__global__ void polar_kernel(int n, const Row *in, Row *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Row r = in[i];
    const double x = hts::double_of(r.b[0]), y = hts::double_of(r.b[1]);
    const hts::RadialBounds rb = hts::radial_bounds(hts::double_of(r.b[2]), hts::double_of(r.b[3]));
    const double n2 = __dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y));
    uint64_t qa = 0, qr = 0;
    Row o;
    o.b[0] = hts::quantise_angle(x, y, 29, qa);
    o.b[2] = hts::quantise_radius(n2, r.b[4] != 0ull, rb, 29, qr);
    o.b[1] = qa;
    o.b[3] = qr;
    o.b[4] = 0;
    out[i] = o;
}

__global__ void math_kernel(int n, const Row *in, Row *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = hts::double_of(in[i].b[0]);
    double t, rs;
    hts::sqrt_rsqrt(x, t, rs);
    out[i] = Row{{hts::bits_of(t), hts::bits_of(rs), hts::bits_of(hts::reciprocal(x)), hts::bits_of(hts::log1p_pos(x)),
                  hts::bits_of(hts::log_pos(x))}};
}

int main(int argc, char **argv)
{
    const bool polar = argc > 1 && !strcmp(argv[1], "polar");
    std::vector<Row> rows;
    Row r{{0, 0, 0, 0, 0}};
    while (polar ? scanf("%llx %llx %llx %llx %llx", r.b, r.b + 1, r.b + 2, r.b + 3, r.b + 4) == 5
                 : scanf("%llx", r.b) == 1)
        rows.push_back(r);
    const int n = (int)rows.size();
    Row *in = nullptr, *out = nullptr;
    if (!n || cudaMalloc(&in, n * sizeof(Row)) != cudaSuccess || cudaMalloc(&out, n * sizeof(Row)) != cudaSuccess) return 1;
    cudaMemcpy(in, rows.data(), n * sizeof(Row), cudaMemcpyHostToDevice);
    if (polar)
        polar_kernel<<<(n + 255) / 256, 256>>>(n, in, out);
    else
        math_kernel<<<(n + 255) / 256, 256>>>(n, in, out);
    if (cudaMemcpy(rows.data(), out, n * sizeof(Row), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    for (const Row &o : rows) printf("%llx %llx %llx %llx %llx\n", o.b[0], o.b[1], o.b[2], o.b[3], o.b[4]);
    return 0;
}
