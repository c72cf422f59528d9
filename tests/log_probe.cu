// The library's double logarithm, for test_log.py.  On the host: log_max_ulp, the largest error of
// the integer path against long double over every interval of the table (edges, middles, both ends of
// the exponents it takes), around 1 and on seeded random arguments.  On the device: log_device, ln_f64
// and CUDA's log of the same arguments.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "fmlbm_log.cuh"

using namespace fmlbm;

static const LogEntry host_table[128] = {FMLBM_LOG_TABLE};

static uint64_t bits_of(double x) {
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
}
static double error_ulp(double x) {
    const uint64_t b = bits_of(x);
    if (!log_reducible(b)) return INFINITY;
    const double got = log_reduced(b, host_table[log_index(b)]);
    const long double want = logl((long double)x);
    if (want == 0.0L) return got == 0.0 ? 0.0 : INFINITY;
    return (double)(fabsl((long double)got - want) / ldexpl(1.0L, ilogbl(want) - 52));
}

extern "C" int log_takes(double x) { return log_reducible(bits_of(x)) ? 1 : 0; }

extern "C" double log_max_ulp(long long randoms, double* worst_at) {
    double worst = 0.0;
    auto look = [&](double x) {
        const double e = error_ulp(x);
        if (!(e <= worst)) {
            worst = e;
            *worst_at = x;
        }
    };
    for (int e = -43; e <= 43; ++e)
        for (int i = 0; i < 128; ++i) {
            // x of exponent e in the binades' 128 equal parts: the table's intervals
            const double lo = ldexp(1.0 + i / 128.0, e), hi = ldexp(1.0 + (i + 1) / 128.0, e);
            look(lo);
            look(nextafter(lo, INFINITY));
            look(0.5 * (lo + hi));
            look(nextafter(nextafter(hi, 0.0), 0.0));
            look(nextafter(hi, 0.0));
        }
    for (int k = 1; k <= 52; ++k)
        for (int m = 0; m < 64; ++m) {
            const double d = ldexp(1.0 + m / 64.0, -k);
            if (1.0 + d < 2.0) look(1.0 + d);
            if (1.0 - d > 0.0) look(1.0 - d);
        }
    uint64_t s = 12345;
    for (long long n = 0; n < randoms; ++n) {
        s += 0x9E3779B97F4A7C15ull;
        uint64_t z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const double u = 1.0 + (double)(z >> 12) * 2.220446049250313e-16;
        // any exponent the path takes, and as often one near 1
        look(ldexp(u, (n & 1) ? (int)(z % 87) - 43 : -(int)(z & 1)));
    }
    return worst;
}

static __global__ void both(const double* x, double* ours, double* cuda, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        ours[i] = ln_f64(x[i]);
        cuda[i] = log(x[i]);
    }
}
// x, ours, cuda: device memory, n values each.
extern "C" int log_device(const double* x, double* ours, double* cuda, int n) {
    both<<<64, 256>>>(x, ours, cuda, n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
