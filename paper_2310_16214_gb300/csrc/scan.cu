// Batched inclusive sum scan (Section III, "Scan Operator"; knobs of
// Section V-B).
//
// One block holds `spb` whole problems of n elements; each problem is served
// by T = n/P threads and each thread owns P consecutive elements, read and
// written with 16-byte streaming accesses.  The prefix is formed in three
// levels:
//   1. thread-serial inclusive scan of the P elements in registers;
//   2. warp-shuffle prefix of the thread totals over aligned segments of
//      min(T, 32) lanes, with the Kogge-Stone or the Ladner-Fischer circuit
//      (Fig. 1(f) / 1(d));
//   3. when T > 32, one shared-memory slot per warp (the 32-slots-per-problem
//      scheme of Section V-B) and a second shuffle prefix over the warp totals.
// int32 arithmetic wraps modulo 2^32, which is exactly the definition.
//
// A length n that is not a power of two runs scan_ragged_kernel with the plan
// of the next power of two n': rows are n apart, elements outside the row
// read as 0 (the identity of the sum) and are not written.
#include "device_util.cuh"
#include "internal.h"

namespace bplg {

// The prefix of one thread's P elements, already summed in v, joined with
// those of the other threads of its problem: tps threads (a power of two up
// to 32, else whole warps), this one in the problem's warp wl.
template <typename E, int P, int PATTERN>
__device__ __forceinline__ void scan_join(E (&v)[P], int tps, int wl, E *warp_tot) {
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int width = tps < 32 ? tps : 32;
    const int lane_in_seg = lane & (width - 1);
    E incl = seg_scan<PATTERN>(v[P - 1], lane_in_seg, width);
    E excl = __shfl_up_sync(kFullMask, incl, 1, width);
    if (lane_in_seg == 0) excl = E(0);

    if (tps > 32) {
        const int warp = tid >> 5;
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        const int wps = tps >> 5;
        E w = (lane < wps) ? warp_tot[(warp - wl) + lane] : E(0);
        w = seg_scan<PATTERN>(w, lane, 32);
        E woff = __shfl_sync(kFullMask, w, wl > 0 ? wl - 1 : 0);
        if (wl == 0) woff = E(0);
        excl += woff;
    }
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] += excl;
}

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
    const int64_t base = sig * n + static_cast<int64_t>(t) * P;

    E v[P];
    if (active) {
        load_run<E, P>(in + base, v);
    } else {
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = E(0);
    }
#pragma unroll
    for (int i = 1; i < P; ++i) v[i] += v[i - 1];
    scan_join<E, P, PATTERN>(v, tps, (tid >> 5) & ((tps >> 5) - 1), warp_tot);
    if (active) store_run<E, P>(out + base, v);
}

// Problems of any length n: as many threads as the row needs (whole warps,
// not the next power of two), elements outside the row read as 0.  A row
// starts at element sig n, which is on a 16-byte boundary only when that is a
// multiple of 4; so the problem begins sh = (sig n) mod 4 zero elements before
// the row, at the boundary, and with P a multiple of 4 every group of 4
// elements wholly inside the row moves as 16 bytes; the at most two others are
// element-wise.  (max_shift 0: no such zeros; rows that start off a
// boundary are element-wise throughout.)
// Measured, n = 5000, 2^24 elements: 320 threads a row instead of 512,
// 0.0307 -> 0.0284 ms; n = 5419 (odd), 1723 rows: 0.0533 -> 0.0185 ms.
template <typename E, int P, int PATTERN>
__global__ void __launch_bounds__(1024)
    scan_ragged_kernel(const E *in, E *out, int tps, int spb, int64_t batch, int64_t n, int max_shift) {
    __shared__ E warp_tot[32];
    using V4 = typename Vec4Of<E>::type;
    constexpr int V = P % 4 == 0 ? 4 : 1;
    const int s = threadIdx.x / tps;
    const int t = threadIdx.x - s * tps;
    const int64_t sig = static_cast<int64_t>(blockIdx.x) * spb + s;
    const bool active = sig < batch;
    const int64_t row0 = sig * n;
    const int sh = static_cast<int>(row0 & max_shift);
    const bool vec = V == 4 && ((row0 - sh) & 3) == 0;
    const int len = static_cast<int>(n), i0 = t * P - sh;  // the thread's first element, as an index of the row
    const int64_t base = row0 + i0;
    E v[P];
#pragma unroll
    for (int q = 0; q < P; q += V) {
        const int i = i0 + q;
        if (vec && active && i >= 0 && i + 3 < len) {
            const V4 w = ld_stream(reinterpret_cast<const V4 *>(in + base + q));
            v[q] = w.x;
            v[q + 1] = w.y;
            v[q + 2] = w.z;
            v[q + 3] = w.w;
        } else {
#pragma unroll
            for (int e = q; e < q + V; ++e) v[e] = active && i0 + e >= 0 && i0 + e < len ? in[base + e] : E(0);
        }
    }
#pragma unroll
    for (int i = 1; i < P; ++i) v[i] += v[i - 1];
    scan_join<E, P, PATTERN>(v, tps, t >> 5, warp_tot);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < P; q += V) {
        const int i = i0 + q;
        if (vec && i >= 0 && i + 3 < len) {
            V4 w;
            w.x = v[q];
            w.y = v[q + 1];
            w.z = v[q + 2];
            w.w = v[q + 3];
            st_stream(reinterpret_cast<V4 *>(out + base + q), w);
        } else {
#pragma unroll
            for (int e = q; e < q + V; ++e)
                if (i0 + e >= 0 && i0 + e < len) out[base + e] = v[e];
        }
    }
}

namespace {

template <typename E, int P, bool RAGGED>
const void *scan_func_p(int pattern) {
    if constexpr (RAGGED)
        return pattern == BPLG_PATTERN_LF ? reinterpret_cast<const void *>(&scan_ragged_kernel<E, P, 1>)
                                          : reinterpret_cast<const void *>(&scan_ragged_kernel<E, P, 0>);
    else
        return pattern == BPLG_PATTERN_LF ? reinterpret_cast<const void *>(&scan_kernel<E, P, 1>)
                                          : reinterpret_cast<const void *>(&scan_kernel<E, P, 0>);
}

template <typename E, bool RAGGED>
const void *scan_func_t(int P, int pattern) {
    switch (P) {
        case 1: return scan_func_p<E, 1, RAGGED>(pattern);
        case 2: return scan_func_p<E, 2, RAGGED>(pattern);
        case 4: return scan_func_p<E, 4, RAGGED>(pattern);
        case 8: return scan_func_p<E, 8, RAGGED>(pattern);
        case 16: return scan_func_p<E, 16, RAGGED>(pattern);
        case 32: return scan_func_p<E, 32, RAGGED>(pattern);
        default: return nullptr;
    }
}

const void *scan_func(int dtype, int P, int pattern, bool ragged) {
    if (dtype == BPLG_I32) return ragged ? scan_func_t<int32_t, true>(P, pattern) : scan_func_t<int32_t, false>(P, pattern);
    if (dtype == BPLG_F32) return ragged ? scan_func_t<float, true>(P, pattern) : scan_func_t<float, false>(P, pattern);
    return nullptr;
}

}  // namespace

bool scan_launch_info(const bplg_plan &p, int dtype, int64_t n, int64_t batch, Launch *out) {
    std::string why;
    if (!plan_structurally_valid(p, dtype, n, &why)) return false;
    const void *f = scan_func(dtype, p.P, p.pattern, false);
    if (!f) return false;
    out->func = f;
    out->threads = p.L;
    out->smem = 0;
    out->blocks = (batch + p.spb - 1) / p.spb;
    return true;
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
        li.func = scan_func(dtype, p.P, p.pattern, true);
        max_shift = p.P % 4 != 0 || n % 4 == 0 ? 0 : (n % 2 == 0 ? 2 : 3);
        const auto threads_for = [&](int64_t len) {
            const int64_t t = (len + p.P - 1) / p.P;
            return static_cast<int>(t <= 32 ? next_pow2(t) : (t + 31) / 32 * 32);
        };
        tps = threads_for(n + max_shift);
        if (spb * tps > 1024) {
            max_shift = 0;
            tps = threads_for(n);
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
