// Mixed-radix Stockham FFT for lengths n = 2^a 3^b 5^c that are not powers
// of two (at most 12288), one kernel per length with its whole stage
// schedule fixed at compile time.  (The paper keeps to N = r^n; this extends
// the radix-r Stockham formulation of Section III to products of small
// radices, so such lengths need not go through Bluestein's identity.)
//
// Stockham autosort, decimation in time.  With n = r_1 r_2 ... r_K, after
// the stages r_1 .. r_{s-1} the array holds, for L = r_1 ... r_{s-1} and
// m = n / L, the L-point DFTs of the m decimated subsequences x[k + m t]
// (t < L): entry j of subsequence k at index j m + k.  Stage s (radix r,
// m' = m / r) joins subsequences k' + m' p (p < r) into the (L r)-point DFT
// of subsequence k': with j'' = j + L q,
//     A'[j + L q][k'] = sum_p W_r^(p q) (W_{L r}^(p j) A[j][k' + m' p]),
// read at j r m' + p m' + k' and written at (j + L q) m' + k'.  After the
// last stage L = n, m = 1 and the array is X in natural order.  W_m =
// exp(dir 2 pi i / m); every stage twiddle W_{L r}^(p j) = W_n^(p j m') comes
// from a table per n (stage_table below), computed on the host in float64
// and rounded to float32, like the power-of-two tables.
//
// Radices 25, 24, 20, 18, 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2: the 3- and 5-point DFTs
// written out, the composite ones as two factors with their inner twiddles
// computed at compile time (float64 series, rounded once).  Because n, the
// radices and every stage's m' are compile-time constants, the index
// arithmetic folds into constants and immediates, and each kernel holds the
// code of its own radices only (so its registers are those of its largest
// codelet).  The plan (kernel_plan below): the fewest stages, radices in
// non-increasing order; T threads per signal, each doing at most B
// butterflies a stage (one in the smallest-radix stage unless n / r_min
// exceeds 1024 threads, or one in the largest-radix stage when the radices
// are at least a factor two apart); S
// signals a block and a register budget, chosen for small blocks and
// enough busy threads per SM.  The signals sit in one shared-memory buffer
// (n complex values each) -- a stage reads its inputs into registers, the
// block waits, and writes its outputs in place -- or in two that the stages
// alternate between, where that costs no block per SM; the first stage
// reads global memory and the last writes it.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <utility>

#include "fft_common.cuh"

namespace bplg {

constexpr int kMixedMaxLen = 12288;  // the largest length with a kernel
constexpr int kMixedShards = 8;      // translation units the kernels are spread over

namespace mixed_detail {

// cos and sin of 2 pi k / m at compile time, in double: the angle is
// reduced exactly (by the quadrant of 4k / m) to [0, pi / 2) and the
// Taylor series of sine and cosine summed there (24 terms: the remainder is
// below 1e-40 for arguments up to pi / 2)
constexpr double kPiD = 3.14159265358979323846264338327950288;
constexpr double taylor_sin(double x) {
    double t = x, sum = x;
    for (int i = 1; i < 24; ++i) {
        t *= -x * x / ((2.0 * i) * (2.0 * i + 1.0));
        sum += t;
    }
    return sum;
}
constexpr double taylor_cos(double x) {
    double t = 1.0, sum = 1.0;
    for (int i = 1; i < 24; ++i) {
        t *= -x * x / ((2.0 * i - 1.0) * (2.0 * i));
        sum += t;
    }
    return sum;
}
constexpr double cos_2pi(int k, int m) {
    const int kk = ((k % m) + m) % m;
    const int q = (4 * kk) / m, r = 4 * kk - q * m;  // angle = (q + r / m) pi / 2
    const double x = 0.5 * kPiD * r / m;
    return q == 0 ? taylor_cos(x) : q == 1 ? -taylor_sin(x) : q == 2 ? -taylor_cos(x) : taylor_sin(x);
}
constexpr double sin_2pi(int k, int m) {
    const int kk = ((k % m) + m) % m;
    const int q = (4 * kk) / m, r = 4 * kk - q * m;
    const double x = 0.5 * kPiD * r / m;
    return q == 0 ? taylor_sin(x) : q == 1 ? taylor_cos(x) : q == 2 ? -taylor_sin(x) : -taylor_cos(x);
}

// In-register 3- and 5-point DFTs, y_q = sum_p v_p exp(DIR 2 pi i p q / R).
// c_k = cos(2 pi k / R), s_k = sin(2 pi k / R).
template <int DIR>
__device__ __forceinline__ void dft3(float2 (&v)[3]) {
    constexpr float c1 = -0.5f, s1 = DIR * 0.86602540378443864676f;
    const float2 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const float2 b = make_float2(fmaf(c1, t.x, v[0].x), fmaf(c1, t.y, v[0].y));
    const float2 e = make_float2(-s1 * d.y, s1 * d.x);  // i s1 d
    v[0] = cadd(v[0], t);
    v[1] = cadd(b, e);
    v[2] = csub(b, e);
}

template <int DIR>
__device__ __forceinline__ void dft5(float2 (&v)[5]) {
    constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    constexpr float s1 = DIR * 0.95105651629515357212f, s2 = DIR * 0.58778525229247312917f;
    const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const float2 d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    const float2 b1 = make_float2(fmaf(c2, t2.x, fmaf(c1, t1.x, v[0].x)), fmaf(c2, t2.y, fmaf(c1, t1.y, v[0].y)));
    const float2 b2 = make_float2(fmaf(c1, t2.x, fmaf(c2, t1.x, v[0].x)), fmaf(c1, t2.y, fmaf(c2, t1.y, v[0].y)));
    // e1 = i (s1 d1 + s2 d2), e2 = i (s2 d1 - s1 d2)
    const float2 u1 = make_float2(fmaf(s2, d2.x, s1 * d1.x), fmaf(s2, d2.y, s1 * d1.y));
    const float2 u2 = make_float2(fmaf(-s1, d2.x, s2 * d1.x), fmaf(-s1, d2.y, s2 * d1.y));
    const float2 e1 = make_float2(-u1.y, u1.x), e2 = make_float2(-u2.y, u2.x);
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = cadd(b1, e1);
    v[4] = csub(b1, e1);
    v[2] = cadd(b2, e2);
    v[3] = csub(b2, e2);
}

template <int R, int DIR>
__device__ __forceinline__ void dft_any(float2 (&v)[R]);

// R = A B points as A B-point DFTs, twiddles W_R^(n1 k2), then B A-point
// DFTs (the two-factor Cooley-Tukey step): with n = n1 + A n2 and
// k = k2 + B k1, X[k] = sum_n1 W_A^(n1 k1) [W_R^(n1 k2) sum_n2 x[n] W_B^(n2 k2)]
template <int A, int B, int DIR>
__device__ __forceinline__ void dft_two_factor(float2 (&v)[A * B]) {
    float2 y[A][B];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
        float2 u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = v[n1 + A * n2];
        dft_any<B, DIR>(u);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            if (n1 == 0 || k2 == 0) {
                y[n1][k2] = u[k2];
            } else {
                const float c = static_cast<float>(cos_2pi(n1 * k2, A * B));
                const float sn = static_cast<float>(DIR * sin_2pi(n1 * k2, A * B));
                y[n1][k2] = make_float2(u[k2].x * c - u[k2].y * sn, u[k2].x * sn + u[k2].y * c);
            }
        }
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        float2 w[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) w[n1] = y[n1][k2];
        dft_any<A, DIR>(w);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[k2 + B * k1] = w[k1];
    }
}

template <int R, int DIR>
__device__ __forceinline__ void dft_any(float2 (&v)[R]) {
    if constexpr (R == 3) {
        dft3<DIR>(v);
    } else if constexpr (R == 5) {
        dft5<DIR>(v);
    } else if constexpr (R == 6) {
        dft_two_factor<2, 3, DIR>(v);
    } else if constexpr (R == 9) {
        dft_two_factor<3, 3, DIR>(v);
    } else if constexpr (R == 10) {
        dft_two_factor<2, 5, DIR>(v);
    } else if constexpr (R == 12) {
        dft_two_factor<4, 3, DIR>(v);
    } else if constexpr (R == 15) {
        dft_two_factor<3, 5, DIR>(v);
    } else if constexpr (R == 18) {
        dft_two_factor<2, 9, DIR>(v);
    } else if constexpr (R == 20) {
        dft_two_factor<4, 5, DIR>(v);
    } else if constexpr (R == 24) {
        dft_two_factor<3, 8, DIR>(v);
    } else if constexpr (R == 25) {
        dft_two_factor<5, 5, DIR>(v);
    } else {
        dft_codelet<R, DIR>(v);
    }
}

// ---------------------------------------------------------------- plan

constexpr int kNumWide = 4;  // the radices above 16, first in the list (kernel_plan)
constexpr int kNumRadices = kNumWide + 11;
constexpr int kRadices[kNumRadices] = {25, 24, 20, 18, 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
constexpr int kMaxStages = 8;
constexpr int kMaxThreads = 1024;
constexpr int kSmemPerSm = 196 * 1024; // shared memory of one SM given to several blocks: beyond it
                                       // 28 KB of L1 are left instead of 60 (at 2^24 points, 228 KB allowed -> this:
                                       // n = 768 0.0584 -> 0.0455 ms, 1600 0.0619 -> 0.0463, 1800 0.0599 -> 0.0512,
                                       // 6561 0.0782 -> 0.0667)
constexpr int kSmemPerBlock = 232448; // the opt-in limit of one block

constexpr bool is_smooth(int n) {
    while (n % 2 == 0) n /= 2;
    while (n % 3 == 0) n /= 3;
    while (n % 5 == 0) n /= 5;
    return n == 1;
}
constexpr bool has_kernel(int n) { return n >= 3 && n <= kMixedMaxLen && (n & (n - 1)) != 0 && is_smooth(n); }

struct Plan {
    int k = 0;                 // stages
    int r[kMaxStages] = {};    // radices, first stage first
    int b = 0;                 // most butterflies a thread does in one stage
    int t = 0;                 // threads per signal
    int spb = 0;               // signals per block
    int threads = 0;           // block size (spb t rounded up to whole warps)
    int minb = 0;              // blocks per SM the register budget is set for
    int vmax = 0;              // complex values a thread holds across a barrier
    bool dbl = false;          // two buffers a signal (one barrier a stage instead of two)
    int pitch[kMaxStages] = {}; // rows of m_s entries that stage s writes, this many places apart
    int sig = 0, sig2 = 0;     // shared-memory places of a signal in its buffer, in the second one
};

// Shared-memory wavefronts of 16 lanes (a half-warp of 8-byte accesses hits 16
// places per wavefront) from lane t0 on, lane t at row t / row, column t % row of
// an array of rows `pitch` places apart.
constexpr int half_warp_wavefronts(int t0, int row, int pitch) {
    int hits[16] = {}, most = 0;
    for (int t = t0; t < t0 + 16; ++t) {
        const int c = ++hits[((t / row) * pitch + t % row) % 16];
        most = c > most ? c : most;
    }
    return most;
}

// Pitch of the rows of m entries between two stages: stage s writes rows of m =
// r' m' (its lanes run along them), stage s + 1, of radix r', reads runs of m' at
// the starts of consecutive rows.  Unpadded, the reads of a short m' fall on few
// banks (rows of 30, runs of 5: three wavefronts for one); the pitch takes the
// fewest wavefronts of both, of equal ones the smallest, and is m unless that
// saves a tenth (n = 4000 gained nothing from 3 %).
constexpr int best_pitch(int m, int m_next) {
    int best = m, best_cost = 1 << 30, plain = 0;
    for (int pitch = m; pitch < m + 16 && (pitch == m || 4 * (pitch - m) <= m); ++pitch) {
        int cost = 0;
        for (int t0 = 0; t0 < 240; t0 += 16)
            cost += half_warp_wavefronts(t0, m, pitch) + half_warp_wavefronts(t0, m_next, pitch);
        if (pitch == m) plain = cost;
        if (cost < best_cost) {
            best = pitch;
            best_cost = cost;
        }
    }
    return 10 * best_cost <= 9 * plain ? best : m;
}

constexpr int rmin_of(const Plan &p) {
    int m = 1 << 30;
    for (int i = 0; i < p.k; ++i) m = p.r[i] < m ? p.r[i] : m;
    return m;
}
constexpr int rmax_of(const Plan &p) {
    int m = 0;
    for (int i = 0; i < p.k; ++i) m = p.r[i] > m ? p.r[i] : m;
    return m;
}
constexpr int bfly_per_thread(int n, int r_min) {
    const int most = n / r_min;  // butterflies of the smallest-radix stage
    return (most + kMaxThreads - 1) / kMaxThreads;
}
// a better than c: fewer stages, then fewer butterflies per thread, then a
// larger smallest radix (stages closer in size, fewer idle threads), then a
// smaller largest radix (smaller codelets)
constexpr bool better(const Plan &a, const Plan &c, int n) {
    if (c.k == 0) return true;
    if (a.k != c.k) return a.k < c.k;
    const int ba = bfly_per_thread(n, rmin_of(a)), bc = bfly_per_thread(n, rmin_of(c));
    if (ba != bc) return ba < bc;
    if (rmin_of(a) != rmin_of(c)) return rmin_of(a) > rmin_of(c);
    return rmax_of(a) < rmax_of(c);
}
constexpr void search(int n, int left, int from, Plan &cur, Plan &best) {
    if (left == 1) {
        if (better(cur, best, n)) best = cur;
        return;
    }
    if (cur.k == kMaxStages || (best.k != 0 && cur.k + 1 > best.k)) return;
    for (int i = from; i < kNumRadices; ++i) {
        if (left % kRadices[i]) continue;
        cur.r[cur.k++] = kRadices[i];
        search(n, left / kRadices[i], i, cur, best);
        --cur.k;
    }
}

constexpr Plan plan_of(int n, int from, bool pad) {
    Plan cur{}, p{};
    search(n, n, from, cur, p);
    const int rmin = rmin_of(p), rmax0 = rmax_of(p);
    auto values = [&](int t) {  // most complex values a thread of t holds in a stage
        int most = 0;
        for (int s = 0; s < p.k; ++s) {
            const int v = (n / p.r[s] + t - 1) / t * p.r[s];
            most = v > most ? v : most;
        }
        return most;
    };
    if (rmax0 >= 2 * rmin && n / rmax0 <= kMaxThreads && (rmax0 < 18 || 4 * values(n / rmax0) <= 5 * rmax0)) {
        // radices at least a factor two apart: one butterfly a thread in the
        // largest-radix stage and several in the smaller-radix ones, rather
        // than idle threads in the large one (measured faster at n = 375,
        // 2000 and 3000; slower at 1620 and 6000, whose radices are closer);
        // above radix 16 only while no stage holds over a quarter more than
        // the largest radix (n = 3200, 20 x 16 x 10, 32 values 0.0615 ms, one
        // butterfly a thread 0.0533; 4000, 20 x 20 x 10, 20 values 0.0527 against 0.0619)
        p.t = n / rmax0;
        p.b = (n / rmin + p.t - 1) / p.t;
    } else {
        p.b = bfly_per_thread(n, rmin);
        p.t = (n / rmin + p.b - 1) / p.b;
    }
    p.vmax = values(p.t);
    // Block shape and register budget.  The budget is at least what the
    // values held across a barrier need (two registers each, plus room for
    // indices, addresses and the codelets' temporaries; 48 for the 12- to
    // 16-point codelets, which need them to keep their loads in flight; 56 from 18 on).
    // Blocks of at most 256 threads where a signal allows: many small blocks, so that one block's barriers stall few
    // threads and the blocks of an SM drift apart, some loading while others
    // compute.  Among the shapes that keep at least 1280 threads (40 warps)
    // of an SM busy, the largest budget (fewer registers cost loads in
    // flight), then the most busy threads, then the fewest signals a block;
    // if no shape reaches that, the most busy threads.
    const int rmax = rmax_of(p);
    int lower = 2 * p.vmax + 12;
    if (lower < 32) lower = 32;
    if (rmax >= 12 && lower < 48) lower = 48;
    if (rmax >= 18 && lower < 56) lower = 56;
    int even = 0, odd = 0;  // places the stages s = 0, 2, .. and 1, 3, .. write
    for (int s = 0, rows = 1; s + 1 < p.k; ++s) {
        rows *= p.r[s];
        p.pitch[s] = pad ? best_pitch(n / rows, n / rows / p.r[s + 1]) : n / rows;
        int &most = s % 2 ? odd : even;
        most = rows * p.pitch[s] > most ? rows * p.pitch[s] : most;
    }
    p.sig = even > odd ? even : odd;
    if (p.sig * 8 > kSmemPerBlock) {  // no room for the padding
        p.sig = even = odd = n;
        for (int s = 0, rows = 1; s + 1 < p.k; ++s) p.pitch[s] = n / (rows *= p.r[s]);
    }
    const int sm1 = p.k > 1 ? p.sig * 8 : 0;
    auto blocks_per_sm = [&](int threads, int smem, int regs) {
        int blocks = 2048 / threads;
        // From radix 15 on a warp's registers are counted in the quarter of the SM
        // they lie in: counted whole, the compiler got 40 registers for a budget of 48
        // and spilled (n = 75 0.0626 -> 0.0556 ms, 240 0.0537 -> 0.0431, 675 0.0731 ->
        // 0.0534; 2304 0.0474 -> 0.0494).  Below, the 40 do, with more warps.
        const int by_regs = rmax >= 15 ? 4 * (512 / ((regs + 7) / 8 * 8)) / (threads / 32)
                                       : 65536 / (threads * ((regs + 7) / 8 * 8));
        if (by_regs < blocks) blocks = by_regs;
        if (smem > 0 && kSmemPerSm / (smem + 1024) < blocks) blocks = kSmemPerSm / (smem + 1024);
        if (blocks > 32) blocks = 32;
        return blocks < 1 ? 1 : blocks;
    };
    constexpr int kBusyTarget = 1280;
    int best_ok = -1, best_regs = 0, best_busy = -1;
    const int max_spb = p.t >= 256 ? 1 : 256 / p.t;
    for (int spb = 1; spb <= max_spb; ++spb) {
        const int threads = (spb * p.t + 31) / 32 * 32;
        if (spb * sm1 > kSmemPerBlock) break;
        // budgets of 64, 56, 48 or 32 registers (at 40 the compiler spilled
        // the 10 x 10 x 10 kernel, slowing it by a fifth)
        for (int regs = 64; regs >= lower || regs == 64; regs -= (regs == 48 ? 16 : 8)) {
            const int r = regs > lower ? regs : lower;
            const int blocks = blocks_per_sm(threads, spb * sm1, r);
            const int busy = blocks * spb * p.t;
            const int ok = busy >= kBusyTarget ? 1 : 0;
            const bool take = ok != best_ok ? ok > best_ok
                              : ok ? (r != best_regs ? r > best_regs : busy > best_busy)
                                   : (busy != best_busy ? busy > best_busy : r > best_regs);
            if (take) {
                best_ok = ok;
                best_regs = r;
                best_busy = busy;
                p.spb = spb;
                p.threads = threads;
                p.minb = blocks;
            }
            if (regs <= lower) break;
        }
    }
    auto blocks_at = [&](int smem) { return blocks_per_sm(p.threads, smem, best_regs); };
    // a second buffer when it costs no block per SM, also where the kernel needs fewer
    // registers than its budget and more blocks are resident than that allows for (n =
    // 216: 32 registers of 48, nine blocks of 22 KB instead of six, 28 KB of L1 left:
    // 0.0577 ms, with one buffer 0.0475; 243 0.0641, 0.0537)
    const int sm2 = (even + odd) * 8;
    p.dbl = p.k > 2 && p.spb * sm2 <= kSmemPerBlock && blocks_at(p.spb * sm2) >= p.minb &&
            blocks_per_sm(p.threads, p.spb * sm2, lower) >= blocks_per_sm(p.threads, p.spb * sm1, lower);
    if (p.dbl) {
        p.sig = even;
        p.sig2 = odd;
    }
    return p;
}

// Shared memory of an SM's blocks, with the 1 KB the system keeps of each.
constexpr int smem_per_sm(const Plan &p) { return p.minb * (p.spb * (p.sig + p.sig2) * 8 + 1024); }

// Padded rows, unless they take a block that fills an SM beyond 196 KB (the next
// size of the shared memory leaves 28 KB of L1 instead of 60, too little for the
// twiddle table: n = 12150 0.106 ms unpadded, 0.113 padded).
constexpr Plan padded_plan(int n, int from) {
    const Plan padded = plan_of(n, from, true);
    if (smem_per_sm(padded) <= kSmemPerSm) return padded;
    const Plan plain = plan_of(n, from, false);
    return smem_per_sm(plain) <= kSmemPerSm ? plain : padded;
}
// The plan with radices up to 16.
constexpr Plan mixed_plan(int n) { return padded_plan(n, kNumWide); }

// The plan of a length's kernel: with radices 25, 24, 20 and 18 too where they save
// a stage, an exchange of every value through shared memory and its barriers (the
// L1 data pipe, 80 % busy, bounds these kernels).  Not up to 288 points, where
// one or two stages of them leave a signal too few threads (n = 24 0.0475 ms with
// radices 6 and 4, 0.111 with one of 24; 288 0.0485 and 0.0573); not with a stage of
// a radix below 9 or a second one less than half the first, whose threads idle in the large
// stage or hold too much in the small ones (1250 0.0576, 0.0627; 2500 0.0593, 0.0658;
// 3125 0.0699, 0.0997); and not where one block is left to an SM instead of several
// (9375 0.0825, 0.0848).  Elsewhere, measured at 2^24 points, radices up to 16 ->
// these: n = 400 0.0595 -> 0.0474 ms, 2000 0.0601 -> 0.0533, 3000 0.0619 -> 0.0557,
// 5120 0.0660 -> 0.0498, 8640 0.103 -> 0.0612, 12000 0.101 -> 0.0829.
constexpr Plan kernel_plan(int n) {
    const Plan narrow = mixed_plan(n), wide = padded_plan(n, 0);
    const bool take = n > 288 && wide.k < narrow.k && wide.r[wide.k - 1] >= 9 && 2 * wide.r[1] >= wide.r[0] &&
                      (wide.minb > 1 || narrow.minb == 1);
    return take ? wide : narrow;
}

constexpr int stage_len_before(const Plan &p, int s) {
    int l = 1;
    for (int i = 0; i < s; ++i) l *= p.r[i];
    return l;
}

// Twiddle table of a length: stage s >= 1 has (r - 1) L entries
// W_n^(p j m), p = 1 .. r - 1, at [stage_table + (p - 1) L + j].  j grows
// with the thread index (by one every m threads), so a warp's loads are
// adjacent or the same; read from one n-point table at p j m they lay up to
// 8 p m bytes apart, a third of the kernel's L1 data-pipe work at n = 3000
// (pipe 80 % busy).  The blocks' sizes telescope: n - r_0 entries in all.
// Measured at 2^24 points: n = 3000 0.0649 -> 0.0614 ms.
constexpr int stage_table(const Plan &p, int s) { return stage_len_before(p, s) - p.r[0]; }

// ---------------------------------------------------------------- kernel

// Stage S: the thread's butterflies b = t + i T (i < B_S), inputs read
// (from global memory in the first stage, else from the shared buffer),
// twiddled and transformed into v[i R + q].
template <int N, int S, int DIR>
__device__ __forceinline__ void stage_in(const float2 *src, const float2 *__restrict__ tw, int t, bool act, bool live,
                                         float2 *v) {
    constexpr Plan P = kernel_plan(N);
    constexpr int R = P.r[S], L = stage_len_before(P, S), m = N / (L * R), nb = N / R;
    constexpr int BS = (nb + P.t - 1) / P.t;
#pragma unroll
    for (int i = 0; i < BS; ++i) {
        const int b = t + i * P.t;
        if (!act || (nb % P.t != 0 && b >= nb)) continue;
        const int j = b / m, k = b - j * m;
        float2 u[R];
#pragma unroll
        for (int p = 0; p < R; ++p) {
            const int e = (S == 0 ? R * j * m : j * P.pitch[S > 0 ? S - 1 : 0]) + k + p * m;
            if constexpr (S == 0)
                u[p] = live ? __ldcs(src + e) : make_float2(0.f, 0.f);
            else
                u[p] = src[e];
        }
        if constexpr (S > 0) {
#pragma unroll
            for (int p = 1; p < R; ++p) {
                float2 w = __ldg(tw + stage_table(P, S) + (p - 1) * L + j);  // W_n^(p j m)
                if (DIR > 0) w.y = -w.y;
                u[p] = cmul(u[p], w);
            }
        }
        dft_any<R, DIR>(u);
#pragma unroll
        for (int q = 0; q < R; ++q) v[i * R + q] = u[q];
    }
}

// Stage S's outputs to the shared buffer, or (LAST) to global memory
template <int N, int S, bool LAST>
__device__ __forceinline__ void stage_out(float2 *dst, int t, bool act, bool live, const float2 *v) {
    constexpr Plan P = kernel_plan(N);
    constexpr int R = P.r[S], L = stage_len_before(P, S), m = N / (L * R), nb = N / R, lm = L * m;
    constexpr int BS = (nb + P.t - 1) / P.t;
#pragma unroll
    for (int i = 0; i < BS; ++i) {
        const int b = t + i * P.t;
        if (!act || (nb % P.t != 0 && b >= nb)) continue;
        const int j = b / m, k = b - j * m;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if constexpr (LAST) {
                if (live) __stcs(dst + j * m + k + q * lm, v[i * R + q]);
            } else {
                dst[j * P.pitch[S] + k + q * (L * P.pitch[S])] = v[i * R + q];
            }
        }
    }
}

// v holds stage S - 1's outputs; write them, then run stage S onwards.
// One buffer: written in place, so every read of a stage is done (a second
// barrier) before its writes.  Two buffers: stage S - 1 writes buffer
// (S - 1) & 1, which nobody reads again before the barrier after stage S's
// writes to the other one.
template <int N, int S, int DIR>
__device__ __forceinline__ void stages_from(float2 *buf, float2 *buf2, float2 *gout, const float2 *__restrict__ tw,
                                            int t, bool act, bool live, float2 *v) {
    constexpr Plan P = kernel_plan(N);
    if constexpr (S == P.k) {
        stage_out<N, S - 1, true>(gout, t, act, live, v);
    } else {
        float2 *cur = P.dbl && ((S - 1) & 1) ? buf2 : buf;
        stage_out<N, S - 1, false>(cur, t, act, live, v);
        __syncthreads();
        stage_in<N, S, DIR>(cur, tw, t, act, live, v);
        if constexpr (!P.dbl && S + 1 < P.k) __syncthreads();
        stages_from<N, S + 1, DIR>(buf, buf2, gout, tw, t, act, live, v);
    }
}

template <int N, int DIR>
__global__ void __launch_bounds__(kernel_plan(N).threads, kernel_plan(N).minb)
    fft_mixed_kernel(const float2 *__restrict__ in, float2 *__restrict__ out, const float2 *__restrict__ tw,
                     int64_t batch) {
    constexpr Plan P = kernel_plan(N);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int s = static_cast<int>(threadIdx.x) / P.t;
    const bool act = s < P.spb;  // threads past spb t (the last warp's tail) only join the barriers
    const int t = static_cast<int>(threadIdx.x) - s * P.t;
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * P.spb + s;
    const bool live = act && sig < batch;
    float2 *buf = reinterpret_cast<float2 *>(smem_raw) + (act ? s : 0) * P.sig;
    float2 *buf2 = P.dbl ? reinterpret_cast<float2 *>(smem_raw) + P.spb * P.sig + (act ? s : 0) * P.sig2 : buf;
    float2 v[P.vmax];
    stage_in<N, 0, DIR>(in + sig * N, tw, t, act, live, v);
    stages_from<N, 1, DIR>(buf, buf2, out + sig * N, tw, t, act, live, v);
}

// ---------------------------------------------------------------- lookup

constexpr int count_lengths() {
    int c = 0;
    for (int n = 3; n <= kMixedMaxLen; ++n) c += has_kernel(n) ? 1 : 0;
    return c;
}
constexpr int kNumLengths = count_lengths();
struct Lengths {
    int v[kNumLengths];
};
constexpr Lengths make_lengths() {
    Lengths l{};
    int c = 0;
    for (int n = 3; n <= kMixedMaxLen; ++n)
        if (has_kernel(n)) l.v[c++] = n;
    return l;
}
constexpr Lengths kLengths = make_lengths();

}  // namespace mixed_detail

struct MixedLaunch {
    const void *fn;
    int threads, spb, smem, stages;
    int radices[mixed_detail::kMaxStages];
};

namespace mixed_detail {

template <int N>
bool fill(int n, int dir, MixedLaunch *o) {
    if (n != N) return false;
    constexpr Plan P = kernel_plan(N);
    o->fn = dir < 0 ? reinterpret_cast<const void *>(&fft_mixed_kernel<N, -1>)
                    : reinterpret_cast<const void *>(&fft_mixed_kernel<N, 1>);
    o->threads = P.threads;
    o->spb = P.spb;
    o->smem = P.k > 1 ? P.spb * (P.sig + P.sig2) * static_cast<int>(sizeof(float2)) : 0;  // one stage: none
    o->stages = P.k;
    for (int i = 0; i < kMaxStages; ++i) o->radices[i] = i < P.k ? P.r[i] : 0;
    return true;
}
template <int K, size_t... I>
bool shard_lookup(int n, int dir, MixedLaunch *o, std::index_sequence<I...>) {
    bool found = false;
    ((found = found || fill<kLengths.v[K + static_cast<int>(I) * kMixedShards]>(n, dir, o)), ...);
    return found;
}

}  // namespace mixed_detail

// The kernels of lengths kLengths.v[K], kLengths.v[K + kMixedShards], ...
// (one translation unit each, compiled in parallel)
template <int K>
bool mixed_shard(int n, int dir, MixedLaunch *o) {
    constexpr int cnt = (mixed_detail::kNumLengths - K + kMixedShards - 1) / kMixedShards;
    return mixed_detail::shard_lookup<K>(n, dir, o, std::make_index_sequence<cnt>{});
}

bool mixed_shard_0(int n, int dir, MixedLaunch *o);
bool mixed_shard_1(int n, int dir, MixedLaunch *o);
bool mixed_shard_2(int n, int dir, MixedLaunch *o);
bool mixed_shard_3(int n, int dir, MixedLaunch *o);
bool mixed_shard_4(int n, int dir, MixedLaunch *o);
bool mixed_shard_5(int n, int dir, MixedLaunch *o);
bool mixed_shard_6(int n, int dir, MixedLaunch *o);
bool mixed_shard_7(int n, int dir, MixedLaunch *o);

}  // namespace bplg
