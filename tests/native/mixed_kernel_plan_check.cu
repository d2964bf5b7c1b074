// Host-side check of the plans the mixed-radix FFT kernels are compiled with
// (kernel_plan of fft_mixed.cuh), built with nvcc and run without a GPU.  For
// every length: radices of the list in non-increasing order that multiply to n,
// no more stages than the plan with radices up to 16; at every exchange the
// writes hit distinct places inside the buffer and the reads find the entry they
// want (run on the kernel's index arithmetic); the block's limits; the twiddle
// blocks fill n - r_0 entries.
#include <cstdio>
#include <vector>

#include "fft_mixed.cuh"

using namespace bplg::mixed_detail;

int main() {
    int count = 0, wide = 0;
    for (int i = 0; i < kNumLengths; ++i) {
        const int n = kLengths.v[i];
        const Plan p = kernel_plan(n);
        auto fail = [&](const char *what, int s) {
            printf("FAIL n=%d stage %d: %s\n", n, s, what);
            return 1;
        };
        long prod = 1;
        for (int s = 0; s < p.k; ++s) {
            bool ok = false;
            for (int r : kRadices) ok = ok || r == p.r[s];
            if (!ok || (s > 0 && p.r[s] > p.r[s - 1])) return fail("radix", s);
            if (p.b * p.t < n / p.r[s]) return fail("butterflies left over", s);
            if ((n / p.r[s] + p.t - 1) / p.t * p.r[s] > p.vmax) return fail("values a thread", s);
            prod *= p.r[s];
        }
        if (prod != n || p.k > mixed_plan(n).k) return fail("product or stages", p.k);
        for (int s = 0; s + 1 < p.k; ++s) {
            const int L = stage_len_before(p, s), m = n / (L * p.r[s]), m2 = m / p.r[s + 1], L2 = L * p.r[s];
            const int size = p.dbl && s % 2 ? p.sig2 : p.sig;
            std::vector<int> at(size, -1);
            for (int b = 0; b < n / p.r[s]; ++b)
                for (int q = 0; q < p.r[s]; ++q) {
                    const int j = b / m, k = b - j * m, e = j * p.pitch[s] + k + q * (L * p.pitch[s]);
                    if (e < 0 || e >= size || at[e] != -1) return fail("write out of place", s);
                    at[e] = (j + L * q) * m + k;
                }
            for (int b = 0; b < n / p.r[s + 1]; ++b)
                for (int q = 0; q < p.r[s + 1]; ++q) {
                    const int j = b / m2, k = b - j * m2, e = j * p.pitch[s] + k + q * m2;
                    if (e < 0 || e >= size || at[e] != j * m + k + q * m2) return fail("read of another entry", s);
                }
            if (stage_table(p, s + 1) + (p.r[s + 1] - 1) * L2 > n - p.r[0]) return fail("twiddle block", s + 1);
        }
        const int smem = p.k > 1 ? p.spb * (p.sig + p.sig2) * 8 : 0;
        if (p.t < 1 || p.spb < 1 || p.threads < p.spb * p.t || p.threads % 32 || p.threads > 1024 ||
            smem > kSmemPerBlock || p.minb < 1 || p.minb * p.threads > 2048)
            return fail("shape", p.k);
        ++count;
        wide += p.r[0] > 16;
    }
    printf("OK %d %d\n", count, wide);
    return wide > 0 ? 0 : 1;
}
