// Host-side check of the run-time planner of the prime-radix FFT
// (fft_prime.cuh), built with nvcc and run without a GPU.  For every length up
// to 12288: a plan exists exactly when the prime factors are at most 31 and not
// all 2, 3 or 5; its radices multiply to n; the block fits the hardware; and over
// every stage of a full block the kernel's divisions by multiplication are
// exact, its reads and writes stay inside the signal (each element written once)
// and its table indices inside the table.  Prints "OK <lengths>" or the first
// failure.
#include <cstdio>
#include <vector>

#include "fft_prime.cuh"

using namespace bplg;

static bool expected(int n) {
    bool large = false;
    for (int q = 2; q <= 31; ++q)
        while (n % q == 0) {
            n /= q;
            large = large || q >= 7;
        }
    return n == 1 && large;
}

int main() {
    int lengths = 0;
    for (int n = 1; n <= kPrimeMaxLen + 1; ++n) {
        const PrimePlan p = prime_plan(n);
        if ((p.stages > 0) != (n <= kPrimeMaxLen && expected(n))) {
            printf("FAIL n=%d: plan with %d stages\n", n, p.stages);
            return 1;
        }
        if (p.stages == 0) continue;
        ++lengths;
        long prod = 1;
        for (int s = 0; s < p.stages; ++s) prod *= p.r[s];
        if (prod != n || prime_smem(p) > 227 * 1024 || p.spb < 1 || p.threads < 64 || p.threads > kPrimeMaxThreads ||
            p.threads % 32 != 0 || p.r[0] < 7) {
            printf("FAIL n=%d: product %ld, %d bytes, spb %d, threads %d\n", n, prod, prime_smem(p), p.spb, p.threads);
            return 1;
        }
        for (int s = 0; s < p.stages; ++s) {
            const int R = p.r[s], L = p.L[s], m = p.m[s], nb = n / R;
            std::vector<char> written(n, 0);
            for (uint32_t i = 0; i < static_cast<uint32_t>(p.spb * nb); ++i) {
                const uint32_t sg = nb > 1 ? static_cast<uint32_t>((uint64_t(i) * p.inv_nb[s]) >> 32) : i;
                const uint32_t b = i - sg * nb, j = m > 1 ? static_cast<uint32_t>((uint64_t(b) * p.inv_m[s]) >> 32) : b;
                bool ok = sg == i / nb && j == b / m;
                for (int q = 0; q < R && ok; ++q) {
                    const int rd = static_cast<int>(b + (R - 1) * j * m + q * m), wr = static_cast<int>(b) + q * L * m;
                    ok = rd >= 0 && rd < n && wr >= 0 && wr < n;
                    if (ok && sg == 0) ok = !written[wr]++;
                    const int tw = L - p.r[0] + (q - 1) * L + static_cast<int>(j);
                    if (s > 0 && q > 0) ok = ok && tw >= 0 && tw < n - p.r[0];
                }
                if (!ok) {
                    printf("FAIL n=%d stage %d butterfly %u\n", n, s, i);
                    return 1;
                }
            }
        }
    }
    printf("OK %d\n", lengths);
    return 0;
}
