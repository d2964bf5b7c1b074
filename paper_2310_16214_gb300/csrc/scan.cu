// Batched inclusive sum scan (Section III, "Scan Operator"; knobs of
// Section V-B).
//
// One block holds `spb` whole problems of n elements; each problem is served
// by T = n/P threads and each thread owns P elements, in rows of four adjacent
// ones (scan_common.cuh), read and written with 16-byte streaming accesses.
// The prefix is formed in three levels:
//   1. thread-serial inclusive scan of each row's elements in registers;
//   2. per row, warp-shuffle prefix of the threads' row totals over aligned
//      segments of min(T, 32) lanes, with the Kogge-Stone or the
//      Ladner-Fischer circuit (Fig. 1(f) / 1(d)); then the rows' sums in order;
//   3. when T > 32, one shared-memory slot per warp (the 32-slots-per-problem
//      scheme of Section V-B) and a second shuffle prefix over the warp totals.
// int32 arithmetic wraps modulo 2^32, which is exactly the definition.
//
// A length n that is not a power of two runs scan_ragged_kernel with the plan
// of the next power of two n': rows are n apart, elements outside the row
// read as 0 (the identity of the sum) and are not written.
#include <algorithm>

#include "device_util.cuh"
#include "internal.h"
#include "scan_common.cuh"

namespace bplg {

template <typename E, int P, int PATTERN, bool RUNS>
__global__ void __launch_bounds__(1024, P <= 8 || (RUNS && P == 16) ? 2 : 1)
    scan_kernel(const E *in, E *out, int log_t, int spb, int64_t batch, int64_t n) {
    __shared__ E warp_tot[32];
    const int tid = threadIdx.x;
    const int tps = 1 << log_t;  // threads per problem
    const int s = tid >> log_t;
    const int t = tid & (tps - 1);
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * spb + s;
    const bool active = sig < batch;
    using S = ScanRows<P, RUNS>;
    constexpr int W = S::W;
    E v[P];
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q) {
        if (active) {
            load_row<E, W>(in + sig * n + S::pos(t, tps, q), v + W * q);
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) v[W * q + i] = E(0);
        }
    }
    scan_problem<E, P, PATTERN, RUNS>(v, tps, (tid >> 5) & ((tps >> 5) - 1), warp_tot);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q) store_row<E, W>(out + sig * n + S::pos(t, tps, q), v + W * q);
}

// Problems of any length n: as many threads as the row needs (whole warps,
// not the next power of two), elements outside the row read as 0.  A row
// starts at element sig n, which is on a 16-byte boundary only when that is a
// multiple of 4; so the problem begins sh = (sig n) mod 4 zero elements before
// the row, at the boundary, and with P a multiple of 4 every group of 4
// elements wholly inside the row moves as 16 bytes; the at most two others are
// element-wise.  (max_shift 0: no such zeros, every access element-wise.)
// Measured at 2^26 elements against the padded power of two's threads with
// element-wise rows: n = 5000 0.109 -> 0.0805 ms, 5001 0.322 -> 0.089, 1100 0.1005
// -> 0.0866, 45 0.136 -> 0.098.
// ALIGNED: n is a multiple of 4, so every row starts on a boundary and a group of
// 4 elements is wholly inside or wholly past it.
// PADDED: 2^threads threads, P consecutive elements each, no zero elements before
// the row.
template <typename E, int P, int PATTERN, bool ALIGNED, bool PADDED>
__global__ void __launch_bounds__(1024, P <= 8 ? 2 : 1)
    scan_ragged_kernel(const E *in, E *out, int threads, int spb, int64_t batch, int64_t n, int max_shift) {
    __shared__ E warp_tot[32];
    using S = ScanRows<P, PADDED>;
    constexpr int W = S::W;
    const int tps = PADDED ? 1 << threads : threads;  // threads per problem
    const int s = PADDED ? threadIdx.x >> threads : (tps <= 32 ? threadIdx.x >> (31 - __clz(tps)) : threadIdx.x / tps);
    const int t = PADDED ? threadIdx.x & (tps - 1) : threadIdx.x - s * tps;
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * spb + s;
    const bool active = sig < batch;
    const int64_t row0 = sig * n;
    const int sh = ALIGNED || PADDED ? 0 : static_cast<int>(row0 & max_shift);
    const bool vec = ALIGNED || (!PADDED && W == 4 && max_shift != 0);  // then row0 - sh is a multiple of 4
    const int len = static_cast<int>(n);
    E v[P];
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q) {
        const int i = S::pos(t, tps, q) - sh;  // the group's first element, as an index of the row
        if (vec && active && (ALIGNED || i >= 0) && i + 3 < len) {
            load_row<E, W>(in + row0 + i, v + W * q);
        } else {
#pragma unroll
            for (int e = 0; e < W; ++e)
                v[W * q + e] = !ALIGNED && active && (PADDED || i + e >= 0) && i + e < len ? in[row0 + i + e] : E(0);
        }
    }
    scan_problem<E, P, PATTERN, PADDED>(v, tps, t >> 5, warp_tot);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q) {
        const int i = S::pos(t, tps, q) - sh;
        if (vec && (ALIGNED || i >= 0) && i + 3 < len) {
            store_row<E, W>(out + row0 + i, v + W * q);
        } else if constexpr (!ALIGNED) {
#pragma unroll
            for (int e = 0; e < W; ++e)
                if ((PADDED || i + e >= 0) && i + e < len) out[row0 + i + e] = v[W * q + e];
        }
    }
}

namespace {

// kernel forms: whole power-of-two problems; any length; any multiple of 4; the
// same in runs (the latter two padded)
enum { kWhole, kRagged, kRagged4, kWholeRuns, kPadded, kPadded4 };

template <typename E, int P, int FORM, int PATTERN>
const void *scan_func_f() {
    constexpr bool runs = FORM >= kWholeRuns;
    if constexpr (FORM == kWhole || FORM == kWholeRuns)
        return reinterpret_cast<const void *>(&scan_kernel<E, P, PATTERN, runs && P >= 16>);
    else
        return reinterpret_cast<const void *>(
            &scan_ragged_kernel<E, P, PATTERN, (FORM == kRagged4 || FORM == kPadded4) && P % 4 == 0, runs>);
}

template <typename E, int FORM>
const void *scan_func_t(int P, int pattern) {
    const bool lf = pattern == BPLG_PATTERN_LF;
    switch (P) {
        case 1: return lf ? scan_func_f<E, 1, FORM, 1>() : scan_func_f<E, 1, FORM, 0>();
        case 2: return lf ? scan_func_f<E, 2, FORM, 1>() : scan_func_f<E, 2, FORM, 0>();
        case 4: return lf ? scan_func_f<E, 4, FORM, 1>() : scan_func_f<E, 4, FORM, 0>();
        case 8: return lf ? scan_func_f<E, 8, FORM, 1>() : scan_func_f<E, 8, FORM, 0>();
        case 16: return lf ? scan_func_f<E, 16, FORM, 1>() : scan_func_f<E, 16, FORM, 0>();
        case 32: return lf ? scan_func_f<E, 32, FORM, 1>() : scan_func_f<E, 32, FORM, 0>();
        default: return nullptr;
    }
}

template <typename E>
const void *scan_func_e(int P, int pattern, int form) {
    switch (form) {
        case kWhole: return scan_func_t<E, kWhole>(P, pattern);
        case kRagged: return scan_func_t<E, kRagged>(P, pattern);
        case kRagged4: return scan_func_t<E, kRagged4>(P, pattern);
        case kWholeRuns: return scan_func_t<E, kWholeRuns>(P, pattern);
        case kPadded: return scan_func_t<E, kPadded>(P, pattern);
        default: return scan_func_t<E, kPadded4>(P, pattern);
    }
}

const void *scan_func(int dtype, int P, int pattern, int form) {
    if (dtype == BPLG_I32) return scan_func_e<int32_t>(P, pattern, form);
    if (dtype == BPLG_F32) return scan_func_e<float>(P, pattern, form);
    return nullptr;
}

}  // namespace

// Whole problems in runs: blocks of 1024 threads with P = 16, of which two fit an SM's
// registers only so (n = 16384 0.0551 ms, in rows 0.0601, 2^25 elements), and one
// thread a problem, which has no lanes to share a row with (P = n = 32: 0.067, 0.072).
bool scan_in_runs(const bplg_plan &p, int64_t n) { return (p.P == 16 && p.L == 1024) || (p.P == 32 && n == 32); }

bool scan_launch_info(const bplg_plan &p, int dtype, int64_t n, int64_t batch, Launch *out) {
    std::string why;
    if (!plan_structurally_valid(p, dtype, n, &why)) return false;
    const void *f = scan_func(dtype, p.P, p.pattern, scan_in_runs(p, n) ? kWholeRuns : kWhole);
    if (!f) return false;
    out->func = f;
    out->threads = p.L;
    out->smem = 0;
    out->blocks = (batch + p.spb - 1) / p.spb;
    return true;
}

// threads of a ragged problem: whole warps, or a power of two inside one
static int ragged_threads(int64_t len, int P) {
    const int64_t t = (len + P - 1) / P;
    return static_cast<int>(t <= 32 ? next_pow2(t) : (t + 31) / 32 * 32);
}

// How a problem of a length that is not a power of two runs under P elements a
// thread of the padded length's plan.
struct RaggedForm {
    bool padded;    // the plan's threads, P consecutive elements each
    int tps;        // threads a problem
    int max_shift;  // elements before a row that share its first 16 bytes, at most
};

// Rows on the threads the length needs, from a 16-byte boundary on, or the padded
// form, whichever measured faster (microseconds, padded / rows, pattern KS, 2^25
// int32 elements unless stated).  Padded:
//   - one thread a problem, on boundaries or below 16 elements (P = 16: n = 12 42 / 45);
//   - P = 8 and 16 on boundaries, n' up to 1024, where a row's four prefixes cost more
//     than its better accesses save (P = 16: n = 300 41 / 52, 640 46 / 54, but 2000 46 /
//     43; P = 8: 160 43 / 48, 400 43 / 46), unless a fifth of the threads goes (P = 8:
//     700 46 / 43) or, at P = 16, the row fills seven eighths of n' (500 84 / 79, 60 84 /
//     78 at 2^26);
//   - P up to 4, where a row is a run, unless a fifth of the threads goes (P = 4: n =
//     130 92 / 97, 257 91 / 78, 511 57 / 68);
//   - P = 8 off boundaries from 33 to 128 elements, less than three quarters of n'
//     (n = 65 58 / 68).
// The elements before a row are left out, and its accesses element-wise, where they
// take a quarter more threads, 16 or more of them (P = 8: n = 127 70 -> 47, 511 57 ->
// 50; at P = 32, 127 takes 8 threads: 79 against 58), and below 16 elements (twice
// the threads: n = 3 0.094 against 0.355 ms at 2^26).
static RaggedForm ragged_form(int64_t n, int P) {
    const int64_t np = next_pow2(n);
    const int t = static_cast<int>(np / P);
    const bool aligned = n % 4 == 0;
    RaggedForm f{};
    f.max_shift = P % 4 != 0 || aligned || n < 16 ? 0 : (n % 2 == 0 ? 2 : 3);
    f.tps = ragged_threads(n + f.max_shift, P);
    const int bare = ragged_threads(n, P);
    if (P >= 8 && f.tps >= 16 && 4 * f.tps > 5 * bare) {
        f.max_shift = 0;
        f.tps = bare;
    }
    const bool fewer = 5 * f.tps <= 4 * t;
    if (P <= 4)
        f.padded = !fewer;
    else if (t == 1)
        f.padded = aligned || n < 16;
    else if (aligned)
        f.padded = P < 32 && np <= 1024 && !fewer && (P == 8 || 8 * n < 7 * np);
    else
        f.padded = P == 8 && (t == 8 || t == 16) && 4 * n < 3 * np;
    if (f.padded) {
        f.max_shift = 0;
        f.tps = t;
    }
    return f;
}

// The plan of a length n that is not a power of two when the caller gives none.
//   - Below 16 elements the accesses are element-wise: P = 4 where that leaves few
//     elements over (7: 0.092 against 0.121 ms at 2^26), else 8 (6: 0.085 against 0.101).
//   - Up to 2^20 elements in all the call is as long as one block: P = 8, the least
//     serial work that 1024 threads allow (16 from n = 8190 on, where the elements before
//     a row would not fit), in blocks of 128 threads or more.  Microseconds on the
//     device at 2^16 elements, P = 8 / 32: n = 800 1.5 / 3.0, 2000 1.9 / 3.3, 5000 2.4 / 3.4.
//   - Multiples of 4 up to 1020: P = 16 from 132 to 380 where n is less than three
//     quarters of n', 32 from 384 to 444 in large batches, else 8 (2^26 int32 elements, P =
//     16 / P = 8 / rows at P = 32: n = 28 84 / 79 / 82 us, 100 80 / 78 / 79, 260 78 / 95 /
//     102, 320 78 / 86 / 88, 400 82 / 83 / 80, 500 84 / 78 / 80, 800 82 / 82 / 80), blocks
//     of 128 threads with P = 8.
//   - Others: the P whose threads are idle least (a row of 1100 elements fills 86 % of
//     the warps it takes at P = 8, 54 % at P = 32: 0.0480 against 0.0585 ms, 2^25
//     elements), the larger one of equals; 32 only from 2^24 elements in all (n = 2000 at
//     2^22 6.0 us, with 16 5.6; 3000 at 2^25 44 us, 46) and where it has the elements before
//     the row (255: 62 us at 2^25, with 16 48), 128 or more off boundaries (65: 0.0607
//     against 0.0580).
// Blocks of about 64 threads otherwise, so that a barrier holds up few.
bplg_plan scan_ragged_plan(int64_t n, int64_t batch) {
    const int64_t np = next_pow2(n);
    const bool small = batch <= (int64_t(1) << 20) / n, large = batch >= (int64_t(1) << 24) / n;
    int best = 8, threads = 64;
    if (n < 16) {
        best = np == 4 || 5 * n > 4 * np ? 4 : 8;
        threads = 128;
    } else if (small) {
        while (best < 32 && (np / best > 1024 || ragged_form(n, best).tps > 1024)) best *= 2;
        threads = 128;
    } else if (n % 4 == 0 && n < 1024) {
        const bool wide = np == 256 || np == 512, full = 4 * n >= 3 * np;
        best = wide && !full ? 16 : (np == 512 && n < 448 && large ? 32 : 8);
        if (best == 8) threads = 128;
    } else {
        double best_use = 0.0;
        for (int P = 32; P >= 8; P /= 2) {
            const RaggedForm f = ragged_form(n, P);
            if (np / P > 1024) continue;
            if (P == 32 && np <= 16384 && (!large || (n % 4 != 0 && (n < 128 || f.max_shift == 0)))) continue;
            const double use = static_cast<double>(n) / (static_cast<double>(P) * f.tps);
            if (use > best_use * 1.05) {
                best = P;
                best_use = use;
            }
        }
    }
    bplg_plan p = {};
    p.op = BPLG_OP_SCAN;
    p.n = static_cast<int32_t>(np);
    p.P = best;
    p.radix = 2;
    p.shuffle = 1;
    p.spb = std::max(1, threads / ragged_form(n, p.P).tps);
    p.L = static_cast<int32_t>(p.spb * (np / p.P));
    plan_finalize(&p, BPLG_I32, np);
    return p;
}

int scan_launch(const bplg_plan &p, int dtype, const void *in, void *out, int64_t n, int64_t batch,
                cudaStream_t s) {
    // a plan made for the next power of two runs a length-n problem padded
    const int64_t np = p.n > 0 ? p.n : n;
    if (np < n || (np != n && np / 2 >= n)) return set_error(BPLG_ERR_INVALID_PLAN, "scan: plan is for another n");
    Launch li;
    if (!scan_launch_info(p, dtype, np, batch, &li)) return set_error(BPLG_ERR_INVALID_PLAN, "scan: plan has no kernel");
    int rc = check_grid(li.blocks, "scan");
    if (rc != BPLG_OK) return rc;
    int log_t = ilog2(np / p.P), spb = p.spb, tps = 0, max_shift = 0;
    if (np != n) {
        // Only n = n' - 1 can need more threads than the plan's; without room for
        // the elements before the row (n = 32767) it goes without them.
        RaggedForm f = ragged_form(n, p.P);
        if (spb * f.tps > 1024) {
            f.max_shift = 0;
            f.tps = ragged_threads(n, p.P);
        }
        li.func = scan_func(dtype, p.P, p.pattern,
                            n % 4 == 0 ? (f.padded ? kPadded4 : kRagged4) : (f.padded ? kPadded : kRagged));
        tps = f.padded ? log_t : f.tps;
        max_shift = f.max_shift;
        li.threads = spb * f.tps;
    }
    void *ragged[] = {const_cast<void **>(&in), &out, &tps, &spb, &batch, &n, &max_shift};
    void *whole[] = {const_cast<void **>(&in), &out, &log_t, &spb, &batch, &n};
    void **args = np != n ? ragged : whole;
    cudaError_t e = cudaLaunchKernel(li.func, dim3(static_cast<unsigned>(li.blocks)), dim3(li.threads), args,
                                     0, s);
    return e == cudaSuccess ? BPLG_OK : cuda_error(e, "scan launch");
}

}  // namespace bplg
