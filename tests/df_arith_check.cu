// recip, divisor_recip and rsqrt_normal (df_arith.cuh) over float64's range against
// 1 / x and long double roots.  Bounds from their series: recip's last operation
// is one multiply-add whose terms are exact to 2^-73 of it, so its error is
// 2^-53 (1 + 2^-8) at most (exponents near the ends: the division itself);
// rsqrt_normal adds to that rounding the one of m r, halved by the series' first
// term, 1.5 x 2^-53, and terms below 2^-60.  Prints "ok <values>".
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "df_arith.cuh"

using namespace signtri;

__global__ void evaluate(int n, const double *x, double *r, double *d, int *ex, double *s)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = recip(x[i]);
    const Divisor<double> v = divisor_recip(x[i]);
    d[i] = v.r;
    ex[i] = v.ex;
    const double a = fabs(x[i]);
    s[i] = a >= 0x1p-1000 && a <= 0x1p1000 ? rsqrt_normal(a) : 0.0;
}

int main()
{
    std::mt19937_64 rng(3);
    std::vector<double> x;
    // every exponent, subnormal ones too, with mantissas at the ends and at random
    for (int e = -1074; e < 1024; e++)
        for (int k = 0; k < 40; k++) {
            const unsigned long long m = k == 0 ? 0 : k == 1 ? (1ull << 52) - 1 : k == 2 ? 1 : k == 3 ? 1ull << 51 : rng() >> 12;
            const double v = std::ldexp(1.0 + (double)m * 0x1p-52, e);
            if (v > 0.0 && std::isfinite(v)) x.push_back(k % 2 ? v : -v);
        }
    const int n = (int)x.size();
    double *dx, *dr, *dd, *ds;
    int *de;
    if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&dr, 8 * n) || cudaMalloc(&dd, 8 * n) || cudaMalloc(&ds, 8 * n) ||
        cudaMalloc(&de, 4 * n))
        return 2;
    cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
    evaluate<<<(n + 255) / 256, 256>>>(n, dx, dr, dd, de, ds);
    std::vector<double> r(n), d(n), s(n);
    std::vector<int> ex(n);
    cudaMemcpy(r.data(), dr, 8 * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(d.data(), dd, 8 * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(s.data(), ds, 8 * n, cudaMemcpyDeviceToHost);
    if (cudaMemcpy(ex.data(), de, 4 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    const long double u = 0x1p-53L;
    for (int i = 0; i < n; i++) {
        const double a = x[i];
        const int e = std::ilogb(a);
        bool ok;
        if (e < 64 - 1023 || e > 1982 - 1023) ok = r[i] == 1.0 / a;
        else ok = fabsl((long double)r[i] * a - 1.0L) <= u * (1.0L + 0x1p-8L);
        // 1 / a = d 2^ex, d a normal number
        ok = ok && std::isnormal(d[i]) &&
             fabsl((long double)d[i] * ldexpl((long double)a, ex[i]) - 1.0L) <= u * (1.0L + 0x1p-8L);
        if (s[i] != 0.0) ok = ok && fabsl(s[i] * sqrtl(fabsl((long double)a)) - 1.0L) <= u * 1.55L;
        if (!ok) {
            std::printf("FAIL x %a recip %a divisor %a 2^%d rsqrt %a\n", a, r[i], d[i], ex[i], s[i]);
            return 1;
        }
    }
    std::printf("ok %d\n", n);
    return 0;
}
