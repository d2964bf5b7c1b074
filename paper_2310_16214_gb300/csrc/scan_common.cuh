// Device code of the batched scan shared by the batched kernels (scan.cu) and
// the uneven-batch kernel: which elements a thread holds, and the prefix over
// a problem.
//
// A thread holds P elements in P / V rows of V = min(P, 4) adjacent ones.  The
// lanes of a warp (or of a problem's tps < 32 threads) are adjacent within a
// row, so every 16-byte access of a warp is 512 contiguous bytes, four
// wavefronts of the L1 data pipe.  (With P consecutive elements a thread the
// lanes lay 4 P bytes apart and an access touched P / 2 lines: at P = 16 the
// pipe was 64 % busy in a kernel that only copies, 19 wavefronts an access.)
// The price is one shuffle prefix per row instead of one per thread, on
// independent rows.  Measured at 2^26 elements, consecutive -> rows (each with
// its best P): n = 4096 0.0867 -> 0.0806 ms, 8192 0.0888 -> 0.0806 (98 % of the copy
// bandwidth), 16384 0.1046 -> 0.0817, 32768 0.156 -> 0.102.
#pragma once

#include "device_util.cuh"

namespace bplg {

// RUNS: P consecutive elements a thread all the same, one prefix for them.
template <int P, bool RUNS = false>
struct ScanRows {
    static constexpr int W = P < 4 ? P : 4;  // elements of one access
    static constexpr int GROUPS = P / W;
    // first element of thread t's access q in its problem of tps threads
    __device__ __forceinline__ static int pos(int t, int tps, int q) {
        if (RUNS || GROUPS == 1) return t * P + q * W;
        return tps >= 32 ? (t >> 5) * (32 * P) + q * (32 * W) + (t & 31) * W : q * (tps * W) + t * W;
    }
};

// The inclusive prefix of a problem whose elements its tps threads hold in v
// as above: a power of two of threads up to 32, else whole warps (wl: this
// thread's warp in the problem).  warp_tot: 32 elements of shared memory.
template <typename E, int P, int PATTERN, bool RUNS = false>
__device__ __forceinline__ void scan_problem(E (&v)[P], int tps, int wl, E *warp_tot) {
    using S = ScanRows<P, RUNS>;
    const int lane = threadIdx.x & 31;
    const int width = tps < 32 ? tps : 32;
    const int lane_in_seg = lane & (width - 1);
    // Every four elements (or fewer) have a prefix of their own and get what is before
    // them in one addition.  (A serial prefix over all of a run of 16 rounded on, at n =
    // 260 to a relative error of 9.5e-8 where this has 7.8e-8.)
    constexpr bool kRuns = RUNS && S::GROUPS > 1;
    E add[S::GROUPS];  // what each four get from those before them
    E off = E(0);      // in the last lane of a segment finally the segment's total
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q) {
        E *g = v + S::W * q;
        if constexpr (kRuns) {  // sums in pairs
            const E cd = g[2] + g[3];
            g[1] += g[0];
            g[2] += g[1];
            g[3] = g[1] + cd;
        } else {
#pragma unroll
            for (int i = 1; i < S::W; ++i) g[i] += g[i - 1];
        }
    }
    if constexpr (kRuns) {
        E run = E(0);  // the run's total after the loop
#pragma unroll
        for (int q = 0; q < S::GROUPS; q += 2) {
            const E g0 = v[S::W * q + S::W - 1], g1 = v[S::W * (q + 1) + S::W - 1];
            add[q] = run;
            add[q + 1] = run + g0;
            run += g0 + g1;
        }
        const E incl = seg_scan<PATTERN>(run, lane_in_seg, width);
        const E excl = __shfl_up_sync(kFullMask, incl, 1, width);
#pragma unroll
        for (int q = 0; q < S::GROUPS; ++q) add[q] += lane_in_seg == 0 ? E(0) : excl;
        off = incl;
    } else {
#pragma unroll
        for (int q = 0; q < S::GROUPS; ++q) {
            const E incl = seg_scan<PATTERN>(v[S::W * q + S::W - 1], lane_in_seg, width);
            const E excl = __shfl_up_sync(kFullMask, incl, 1, width);
            add[q] = off + (lane_in_seg == 0 ? E(0) : excl);
            off += q + 1 < S::GROUPS ? __shfl_sync(kFullMask, incl, width - 1, width) : incl;
        }
    }
    if (tps > 32) {
        const int warp = threadIdx.x >> 5;
        if (lane == 31) warp_tot[warp] = off;
        __syncthreads();
        const int wps = tps >> 5;
        E w = (lane < wps) ? warp_tot[(warp - wl) + lane] : E(0);
        w = seg_scan<PATTERN>(w, lane, 32);
        E before = __shfl_sync(kFullMask, w, wl > 0 ? wl - 1 : 0);
        if (wl == 0) before = E(0);
#pragma unroll
        for (int q = 0; q < S::GROUPS; ++q) add[q] += before;
    }
#pragma unroll
    for (int q = 0; q < S::GROUPS; ++q)
#pragma unroll
        for (int i = 0; i < S::W; ++i) v[S::W * q + i] += add[q];
}

// One access of a thread: V elements at p, aligned to V elements.
template <typename E, int V>
__device__ __forceinline__ void load_row(const E *p, E *v) {
    E r[V];
    load_run<E, V>(p, r);
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = r[i];
}
template <typename E, int V>
__device__ __forceinline__ void store_row(E *p, const E *v) {
    E r[V];
#pragma unroll
    for (int i = 0; i < V; ++i) r[i] = v[i];
    store_run<E, V>(p, r);
}

}  // namespace bplg
