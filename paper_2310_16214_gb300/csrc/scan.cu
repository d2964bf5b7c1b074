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

template <typename E, int P, int PATTERN>
__global__ void __launch_bounds__(1024)
    scan_kernel(const E *in, E *out, int log_t, int spb, int64_t batch, int64_t n) {
    __shared__ E warp_tot[32];
    const int tid = threadIdx.x;
    const int tps = 1 << log_t;  // threads per problem
    const int s = tid >> log_t;
    const int t = tid & (tps - 1);
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * spb + s;
    const bool active = sig < batch;
    using S = ScanRows<P>;
    E v[P];
#pragma unroll
    for (int q = 0; q < S::ROWS; ++q) {
        if (active) {
            load_row<E, S::V>(in + sig * n + S::pos(t, tps, q), v + S::V * q);
        } else {
#pragma unroll
            for (int i = 0; i < S::V; ++i) v[S::V * q + i] = E(0);
        }
    }
    scan_problem<E, P, PATTERN>(v, tps, (tid >> 5) & ((tps >> 5) - 1), warp_tot);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < S::ROWS; ++q) store_row<E, S::V>(out + sig * n + S::pos(t, tps, q), v + S::V * q);
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
template <typename E, int P, int PATTERN, bool ALIGNED>
__global__ void __launch_bounds__(1024)
    scan_ragged_kernel(const E *in, E *out, int tps, int spb, int64_t batch, int64_t n, int max_shift) {
    __shared__ E warp_tot[32];
    using S = ScanRows<P>;
    const int s = tps <= 32 ? threadIdx.x >> (31 - __clz(tps)) : threadIdx.x / tps;  // a power of two up to 32
    const int t = threadIdx.x - s * tps;
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * spb + s;
    const bool active = sig < batch;
    const int64_t row0 = sig * n;
    const int sh = ALIGNED ? 0 : static_cast<int>(row0 & max_shift);
    const bool vec = ALIGNED || (S::V == 4 && max_shift != 0);  // then row0 - sh is a multiple of 4
    const int len = static_cast<int>(n);
    E v[P];
#pragma unroll
    for (int q = 0; q < S::ROWS; ++q) {
        const int i = S::pos(t, tps, q) - sh;  // the row's first element, as an index of the problem
        if (vec && active && i >= 0 && i + 3 < len) {
            load_row<E, S::V>(in + row0 + i, v + S::V * q);
        } else {
#pragma unroll
            for (int e = 0; e < S::V; ++e)
                v[S::V * q + e] = !ALIGNED && active && i + e >= 0 && i + e < len ? in[row0 + i + e] : E(0);
        }
    }
    scan_problem<E, P, PATTERN>(v, tps, t >> 5, warp_tot);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < S::ROWS; ++q) {
        const int i = S::pos(t, tps, q) - sh;
        if (vec && i >= 0 && i + 3 < len) {
            store_row<E, S::V>(out + row0 + i, v + S::V * q);
        } else if constexpr (!ALIGNED) {
#pragma unroll
            for (int e = 0; e < S::V; ++e)
                if (i + e >= 0 && i + e < len) out[row0 + i + e] = v[S::V * q + e];
        }
    }
}

namespace {

// kernel forms: whole power-of-two problems, any length, any multiple of 4
enum { kWhole, kRagged, kRagged4 };

template <typename E, int P, int FORM, int PATTERN>
const void *scan_func_f() {
    if constexpr (FORM == kWhole)
        return reinterpret_cast<const void *>(&scan_kernel<E, P, PATTERN>);
    else
        return reinterpret_cast<const void *>(&scan_ragged_kernel<E, P, PATTERN, FORM == kRagged4 && P % 4 == 0>);
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
    return form == kWhole ? scan_func_t<E, kWhole>(P, pattern)
                          : (form == kRagged ? scan_func_t<E, kRagged>(P, pattern) : scan_func_t<E, kRagged4>(P, pattern));
}

const void *scan_func(int dtype, int P, int pattern, int form) {
    if (dtype == BPLG_I32) return scan_func_e<int32_t>(P, pattern, form);
    if (dtype == BPLG_F32) return scan_func_e<float>(P, pattern, form);
    return nullptr;
}

}  // namespace

bool scan_launch_info(const bplg_plan &p, int dtype, int64_t n, int64_t batch, Launch *out) {
    std::string why;
    if (!plan_structurally_valid(p, dtype, n, &why)) return false;
    const void *f = scan_func(dtype, p.P, p.pattern, kWhole);
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

// elements before a row of length n that share its first 16 bytes, at most; rows
// of fewer than 16 stay element-wise (they would take twice the threads: n = 3
// 0.094 against 0.355 ms)
static int ragged_shift(int64_t n, int P) {
    return P % 4 != 0 || n % 4 == 0 || n < 16 ? 0 : (n % 2 == 0 ? 2 : 3);
}

// The plan of a length n that is not a power of two when the caller gives none:
// the P whose threads are idle least (a row of 1100 elements fills 86 % of the
// warps it takes at P = 8, 54 % at P = 32: 0.0480 against 0.0585 ms, 2^25
// elements), the larger one of equals (300: 0.0497 ms at P = 32, 0.0524 at 16,
// 0.0591 at 8), but 16 below 64 (24: 0.0783 against 0.0947 at 2^26) and for
// rows off boundaries below 128 (65: 0.0580 against 0.0607), and at least 8
// (260: 0.0544 at 32, 0.0709 at 4 with fewer threads idle).  Below 16 the
// accesses are element-wise: P = 4 where that leaves few elements over (7: 0.092
// against 0.121 at 2^26), else 8 (6: 0.085 against 0.101).  Blocks of about 64
// threads (128 below 16), so that a barrier holds up few.
bplg_plan scan_ragged_plan(int64_t n) {
    const int64_t np = next_pow2(n);
    int best = n < 16 && (np == 4 || 5 * n > 4 * np) ? 4 : 8;
    double best_use = 0.0;
    for (int P = 32; P >= 8 && n >= 16; P /= 2) {
        if (np / P > 1024 || (P == 32 && n < (n % 4 == 0 ? 64 : 128))) continue;
        const double use = static_cast<double>(n) / (static_cast<double>(P) * ragged_threads(n + ragged_shift(n, P), P));
        if (use > best_use * 1.05) {
            best = P;
            best_use = use;
        }
    }
    bplg_plan p = {};
    p.op = BPLG_OP_SCAN;
    p.n = static_cast<int32_t>(np);
    p.P = best;
    p.radix = 2;
    p.shuffle = 1;
    p.spb = std::max(1, (n < 16 ? 128 : 64) / ragged_threads(n + ragged_shift(n, p.P), p.P));
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
    int log_t = ilog2(np / p.P), spb = p.spb;
    int tps = 1 << log_t, max_shift = 0;
    if (np != n) {
        // threads for the row and the elements before it up to a 16-byte
        // boundary (at most 2 when n is even, 3 when odd): whole warps, or a
        // power of two inside one.  Only n = n' - 1 can need more than the
        // plan's; without room for them (n = 32767) there is no shift.
        li.func = scan_func(dtype, p.P, p.pattern, n % 4 == 0 ? kRagged4 : kRagged);
        max_shift = ragged_shift(n, p.P);
        tps = ragged_threads(n + max_shift, p.P);
        if (spb * tps > 1024) {
            max_shift = 0;
            tps = ragged_threads(n, p.P);
        }
        li.threads = spb * tps;
    }
    void *ragged[] = {const_cast<void **>(&in), &out, &tps, &spb, &batch, &n, &max_shift};
    void *whole[] = {const_cast<void **>(&in), &out, &log_t, &spb, &batch, &n};
    void **args = np != n ? ragged : whole;
    cudaError_t e = cudaLaunchKernel(li.func, dim3(static_cast<unsigned>(li.blocks)), dim3(li.threads), args,
                                     0, s);
    return e == cudaSuccess ? BPLG_OK : cuda_error(e, "scan launch");
}

}  // namespace bplg
