// Mixed-radix Stockham FFT with prime radices 7 to 31, for the lengths whose
// prime factors are at most 31 and not all 2, 3 or 5 (those have the
// compile-time kernels of fft_mixed.cuh); n <= 12288.  Same decimation-in-time
// stages, indices and twiddle table as there, planned at run time, because such
// lengths are too many for a kernel each.
#pragma once

#include <stdint.h>

#include <initializer_list>

namespace bplg {

constexpr int kPrimeMaxLen = 12288;
constexpr int kPrimeMaxStages = 8;
constexpr int kPrimeMaxThreads = 256;

struct PrimePlan {
    int n = 0, stages = 0;                   // points, stages
    int spb = 0, threads = 0;                // signals and threads per block
    int r[kPrimeMaxStages] = {};             // radices, the largest prime first
    int L[kPrimeMaxStages] = {};             // product of the radices before
    int m[kPrimeMaxStages] = {};             // n / (L r)
    uint32_t inv_m[kPrimeMaxStages] = {};    // ceil(2^32 / m), m > 1
    uint32_t inv_nb[kPrimeMaxStages] = {};   // ceil(2^32 / (n / r)), n > r
};

// floor(x / d) from inv = ceil(2^32 / d): exact for x d < 2^32 and d > 1
// (inv d - 2^32 < d, so the error x (inv d - 2^32) / (d 2^32) stays below 1 / d)
inline uint32_t prime_inverse(int d) { return d > 1 ? static_cast<uint32_t>(((uint64_t(1) << 32) + d - 1) / d) : 0u; }

inline int prime_smem(const PrimePlan &p) { return p.stages > 1 ? 2 * p.spb * p.n * 8 : 0; }

// registers of the kernel that serves lengths up to this prime (fft_prime.cu)
inline int prime_tier(int largest) { return largest <= 13 ? 13 : (largest <= 19 ? 19 : 31); }
inline int prime_regs(int tier) { return tier == 13 ? 64 : (tier == 19 ? 80 : 128); }

// Block shape: the threads (64, 128 or 256) and signals per block with the least
// estimated time per signal.  A stage of radix r takes ceil(spb (n / r) / threads)
// rounds of one butterfly a thread, of which the last is often nearly empty (n = 899
// = 31 * 29 with 256 threads and 2 signals: 62 butterflies a stage); the SM runs as
// many blocks as registers and shared memory allow, and from about 1024 threads on
// more of them no longer shorten the time.  One stage (n a prime): 256 threads,
// about 2048 points.
inline void prime_shape(PrimePlan *p) {
    const int regs = prime_regs(prime_tier(p->r[0]));
    double best = 0.0;
    if (p->stages == 1) {
        p->threads = 256;
        p->spb = 2048 / p->n;
        return;
    }
    for (int threads = 64; threads <= kPrimeMaxThreads; threads *= 2)
        for (int spb = 1; spb == 1 || (spb * p->n <= 4096 && spb <= 512); ++spb) {
            PrimePlan q = *p;
            q.spb = spb;
            int blocks = 65536 / (regs * threads), by_smem = prime_smem(q) > 0 ? 232448 / (prime_smem(q) + 1024) : blocks;
            if (by_smem < blocks) blocks = by_smem;
            if (blocks > 32) blocks = 32;
            if (blocks < 1) continue;
            double cost = 0.0;  // of a block, in instructions of a thread
            for (int s = 0; s < p->stages; ++s) {
                const int r = p->r[s], rounds = (spb * (p->n / r) + threads - 1) / threads;
                cost += rounds * (60.0 + 14.0 * r + (r >= 7 && r % 2 == 1 && r != 9 ? 1.0 * r * r : 4.0 * r)) + 60.0;
            }
            const double busy = blocks * threads / 1024.0;
            cost *= (busy > 1.0 ? busy : 1.0) / (static_cast<double>(blocks) * spb);
            if (best == 0.0 || cost < best) {
                best = cost;
                p->spb = spb;
                p->threads = threads;
            }
        }
}

// The plan of n, stages = 0 where n has none.  The primes from 7 on are stages of
// their own, largest first; what is left, 2^a 3^b 5^c, takes the fewest radices of
// 10, 9, 8, 6, 5, 4, 3, 2, of equal choices the one whose smallest is largest.
inline PrimePlan prime_plan(int64_t n) {
    PrimePlan p;
    if (n < 7 || n > kPrimeMaxLen) return p;
    int rest = static_cast<int>(n), k = 0, r[32];
    for (int q : {31, 29, 23, 19, 17, 13, 11, 7})
        while (rest % q == 0) {
            r[k++] = q;
            rest /= q;
        }
    if (k == 0) return p;  // a product of 2, 3 and 5, or of larger primes
    const int smooth[] = {10, 9, 8, 6, 5, 4, 3, 2};
    // depth first in decreasing order
    int best[32], nbest = 32, cur[32];
    struct Search {
        static void run(const int *s, int left, int from, int *cur, int depth, int *best, int &nbest) {
            if (left == 1) {
                if (depth < nbest || (depth == nbest && cur[depth - 1] > best[depth - 1])) {
                    nbest = depth;
                    for (int i = 0; i < depth; ++i) best[i] = cur[i];
                }
                return;
            }
            if (depth >= nbest) return;
            for (int i = from; i < 8; ++i)
                if (left % s[i] == 0) {
                    cur[depth] = s[i];
                    run(s, left / s[i], i, cur, depth + 1, best, nbest);
                }
        }
    };
    Search::run(smooth, rest, 0, cur, 0, best, nbest);
    if (nbest == 32 || k + nbest > kPrimeMaxStages) return p;  // a prime factor above 31
    for (int i = 0; i < nbest; ++i) r[k++] = best[i];
    p.n = static_cast<int>(n);
    p.stages = k;
    int L = 1;
    for (int s = 0; s < k; ++s) {
        p.r[s] = r[s];
        p.L[s] = L;
        p.m[s] = p.n / (L * r[s]);
        p.inv_m[s] = prime_inverse(p.m[s]);
        p.inv_nb[s] = prime_inverse(p.n / r[s]);
        L *= r[s];
    }
    prime_shape(&p);
    return p;
}

}  // namespace bplg
