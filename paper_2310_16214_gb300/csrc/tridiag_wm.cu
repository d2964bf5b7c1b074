// Batched tridiagonal solver by divide and conquer in the manner of Wang and
// Mou (Section III lists it among BPLG's solvers, Fig. 1(e) draws its
// prefix pattern; Section V-A notes it is the solver whose radix can be
// tuned).  Equation i is a_i x_{i-1} + b_i x_i + c_i x_{i+1} = d_i with
// x_{-1} = x_n = 0.
//
// A run of consecutive equations [l, h] fixes its unknowns once the two
// unknowns just outside it, X = x_{l-1} and Y = x_{h+1}, are given; by
// linearity every unknown of the run is an affine function of them,
//     x_i = alpha_i + beta_i X + gamma_i Y.
// The method starts from short runs and repeatedly merges r adjacent runs
// into one, re-expressing the unknowns in terms of the merged run's outer
// neighbours, until one run covers the system; there X = Y = 0 and
// x_i = alpha_i.
//
// Merging r runs.  Let u_k be the last unknown of run k and v_k the first
// unknown of run k+1 (k = 0 .. r-2).  Run k's descriptor gives u_k in terms
// of its own neighbours u_{k-1} (X for k = 0) and v_k, and run k+1's gives
// v_k in terms of u_k and v_{k+1} (Y for k = r-2).  A forward sweep writes
// u_k = p_k + q_k X + s_k v_k; a backward sweep from v_{r-1} = Y then gives
// every v_k and u_k as affine functions of (X, Y).  Both sweeps share the
// pivots 1 - s_k F_{k+1}.x, which stay in (0, 2) for a strictly diagonally
// dominant matrix (every |beta| + |gamma| < 1 there).
//
// GB300 mapping.  Thread t of a system owns P consecutive equations.
//  (1) It computes alpha, beta, gamma of its own run in registers with one
//      Thomas sweep for three right-hand sides (d; -a_first at the first row;
//      -c_last at the last row).
//  (2) Merge stages of radix r (the `radix` knob) combine the threads' runs.
//      Only the first and last unknown of each thread's run are carried
//      through the stages (six numbers per thread).  A stage needs from each
//      of the r runs of its group the run's first and last descriptors; they
//      come by warp shuffles while a group fits in a warp (`shuffle` knob)
//      and through shared memory otherwise (one barrier per stage, double
//      buffered).
//  (3) Once the system is one run, each thread's first and last unknowns
//      are known; the interior ones follow from the thread's own alpha,
//      beta, gamma and its neighbours' boundary values.  The method's
//      stage-by-stage re-expression of the interior unknowns is applied once
//      at the end instead, which gives the same values in exact arithmetic.
// Divisions use the hardware reciprocal (about 1 ulp), as in the CR solver.
#include <string>

#include "device_util.cuh"
#include "internal.h"
#include "tma.cuh"
#include "tridiag_common.cuh"
#include "tridiag_wm.cuh"

namespace bplg {

namespace {

using wm::wm_warp_only;

// RAGGED: systems of nrow < 2^logn equations (rows nrow apart), solved as
// the power-of-two system padded with identity rows (a = c = 0, b = 1,
// d = 0, whose unknowns are 0); c of the last real row is taken as 0 and
// nothing past nrow is read or written.  Accesses are 16 bytes wide when
// nrow is a multiple of 4 and P of 4, else element-wise.
template <int P, int R, int SHUFFLE, int MAXT, bool RAGGED>
__global__ void __launch_bounds__(MAXT)
    tridiag_wm_kernel(const float *ga, const float *gb, const float *gc, const float *gd, float *x, int logn,
                      int log_tps, int spb, int64_t batch, int nrow) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int s = threadIdx.x >> log_tps;
    const int t = threadIdx.x & ((1 << log_tps) - 1);
    const int64_t sig0 = static_cast<int64_t>(blockIdx.x) * spb;
    const int64_t left = batch - sig0;
    const int nvalid = left < spb ? static_cast<int>(left) : spb;
    const bool active = s < nvalid;
    float4 *buf = reinterpret_cast<float4 *>(smem_raw);
    if constexpr (!RAGGED) {
        const int64_t g0 = (sig0 + s) * (int64_t(1) << logn) + static_cast<int64_t>(t) * P;
        wm::wm_solve<P, R, SHUFFLE>(ga + g0, gb + g0, gc + g0, gd + g0, x + g0, active, log_tps, buf);
    } else {
        const int i0 = t * P;
        const int64_t g0 = (sig0 + s) * static_cast<int64_t>(nrow) + i0;
        float a[P], b[P], c[P], d[P];
        // nrow a multiple of 4: rows start on 16-byte boundaries and a group of
        // 4 equations is wholly inside or wholly past the system
        const bool vec4 = P % 4 == 0 && (nrow & 3) == 0;
        if (vec4) {
#pragma unroll
            for (int q = 0; q < (P >= 4 ? P / 4 : 0); ++q) {
                const bool in = active && i0 + 4 * q < nrow;
                float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = make_float4(1.f, 1.f, 1.f, 1.f), vc = va, vd = va;
                if (in) {
                    va = __ldcs(reinterpret_cast<const float4 *>(ga + g0) + q);
                    vb = __ldcs(reinterpret_cast<const float4 *>(gb + g0) + q);
                    vc = __ldcs(reinterpret_cast<const float4 *>(gc + g0) + q);
                    vd = __ldcs(reinterpret_cast<const float4 *>(gd + g0) + q);
                }
                a[4 * q] = va.x; a[4 * q + 1] = va.y; a[4 * q + 2] = va.z; a[4 * q + 3] = va.w;
                b[4 * q] = vb.x; b[4 * q + 1] = vb.y; b[4 * q + 2] = vb.z; b[4 * q + 3] = vb.w;
                c[4 * q] = vc.x; c[4 * q + 1] = vc.y; c[4 * q + 2] = vc.z; c[4 * q + 3] = vc.w;
                d[4 * q] = vd.x; d[4 * q + 1] = vd.y; d[4 * q + 2] = vd.z; d[4 * q + 3] = vd.w;
            }
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (i0 + i == nrow - 1) c[i] = 0.f;  // the last row's c is outside the matrix
        } else {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const bool in = active && i0 + i < nrow;
                a[i] = in ? ga[g0 + i] : 0.f;
                b[i] = in ? gb[g0 + i] : 1.f;
                c[i] = active && i0 + i < nrow - 1 ? gc[g0 + i] : 0.f;
                d[i] = in ? gd[g0 + i] : 0.f;
            }
        }
        const int nval = nrow - i0 < 0 ? 0 : (nrow - i0 < P ? nrow - i0 : P);
        wm::wm_solve_regs<P, R, SHUFFLE>(a, b, c, d, x + g0, active && nval > 0, log_tps, buf, nval, vec4);
    }
}

// Systems of a length that is not a power of two without a plan, from a
// persistent grid, one system per block at a time: the four coefficient rows
// arrive in shared memory by bulk copies (from the 16-byte boundary before the
// row to the one after it), each thread takes its P equations into registers, and
// the slot is refilled with the block's next system while this one is solved
// and stored, so HBM reads go on throughout.
//   Layout.  Threads that read P consecutive equations straight from global
// memory are 4 P bytes apart, and a 16-byte load of a warp then touches P / 2
// lines: at P = 16 (n = 3000) the loads and stores were most of the work of the
// L1 data pipe (57 % busy at 23 % occupancy), and rows off a 16-byte boundary had
// to be read element by element.  From shared memory with P = 12 or 20 the lanes
// lie 3 or 5 16-byte units apart, an odd number, so the eight lanes of each
// phase hit distinct banks and a load takes the least four wavefronts; and the
// row may start anywhere (sh elements of the copy precede it).
//   Threads.  The tps threads the row needs, in whole warps: those missing from
// the merge tree stand for identity rows, whose descriptors are zero, which is
// what their shared-memory slots hold.  PER_WARP (one exchange slot a warp) lets
// two blocks of 98 KB fit where one slot a thread takes 118 KB: n = 5000 0.085 ->
// 0.071 ms; below that it only adds shuffles (0.0594 -> 0.0615 ms at n = 3000).
//   Measured at 2^24 unknowns, padded power-of-two kernel -> this one: n = 300
// 0.076 -> 0.062 ms, 700 0.072 -> 0.062, 1500 0.066 -> 0.055, 3000 0.086 -> 0.060 (82
// % of the copy bandwidth), 3001 0.182 -> 0.060, 5000 0.124 -> 0.065, 8191 0.195 ->
// 0.076.
template <int P, int MAXT, int MINB, bool PER_WARP>
__global__ void __launch_bounds__(MAXT, MINB)
    tridiag_wm_tma_kernel(const float *ga, const float *gb, const float *gc, const float *gd, float *x, int log_tps,
                          int64_t batch, int nrow) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full;
    const int tps = blockDim.x, t = threadIdx.x;
    constexpr int W = PER_WARP ? 5 : 0;  // log2 of the threads that share an exchange slot
    const int slots = (1 << log_tps) >> W, len = tps * P;
    float4 *buf = reinterpret_cast<float4 *>(smem_raw);
    float *slot = reinterpret_cast<float *>(buf + 4 * slots);  // a, b, c, d, `len` floats each
    const int64_t total = batch * nrow;
    // elements copied of a row that starts at row0: whole 16-byte units, and not past
    // the end of the arrays (the last row's last elements are then read directly)
    auto copied = [&](int64_t row0) {
        const int sh = static_cast<int>(row0 & 3);
        const int count = (sh + nrow + 3) & ~3;
        return row0 - sh + count > total ? count - 4 : count;
    };
    auto issue = [&](int64_t sys) {
        const int64_t row0 = sys * nrow;
        const uint32_t bytes = static_cast<uint32_t>(copied(row0)) * 4u;
        const int64_t from = row0 - (row0 & 3);
        mbar_arrive_expect_tx(&full, 4 * bytes);
        tma_load_1d(slot, ga + from, bytes, &full);
        tma_load_1d(slot + len, gb + from, bytes, &full);
        tma_load_1d(slot + 2 * len, gc + from, bytes, &full);
        tma_load_1d(slot + 3 * len, gd + from, bytes, &full);
    };
    if (t == 0) {
        mbar_init(&full, 1);
        fence_mbar_init();
        issue(blockIdx.x);
    }
    const int absent = slots - (tps >> W);  // the absent threads' descriptors
    for (int k = t; k < 4 * absent; k += tps)
        buf[(k / absent) * slots + (tps >> W) + k % absent] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    uint32_t parity = 0;
    for (int64_t sys = blockIdx.x; sys < batch; sys += gridDim.x, parity ^= 1u) {
        const bool ok = mbar_wait_block(&full, parity, t == 0);
        float a[P], b[P], c[P], d[P];
        const float4 *s4 = reinterpret_cast<const float4 *>(slot + t * P);
#pragma unroll
        for (int q = 0; q < P / 4; ++q) {
            const float4 va = s4[q], vb = s4[len / 4 + q], vc = s4[2 * (len / 4) + q], vd = s4[3 * (len / 4) + q];
            a[4 * q] = va.x; a[4 * q + 1] = va.y; a[4 * q + 2] = va.z; a[4 * q + 3] = va.w;
            b[4 * q] = vb.x; b[4 * q + 1] = vb.y; b[4 * q + 2] = vb.z; b[4 * q + 3] = vb.w;
            c[4 * q] = vc.x; c[4 * q + 1] = vc.y; c[4 * q + 2] = vc.z; c[4 * q + 3] = vc.w;
            d[4 * q] = vd.x; d[4 * q + 1] = vd.y; d[4 * q + 2] = vd.z; d[4 * q + 3] = vd.w;
        }
        // the slot is read (and the exchange buffers of the last system too)
        if (!__syncthreads_and(ok)) return;  // a wait ran out; thread 0 has waited again
        if (t == 0 && sys + gridDim.x < batch) {
            fence_proxy_async();
            issue(sys + gridDim.x);
        }
        const int64_t row0 = sys * nrow;
        const int sh = static_cast<int>(row0 & 3);
        const int i0 = t * P - sh;  // the thread's first equation, as an index of the row
        if (i0 <= 0 || i0 + P >= nrow) {
            // the first and the last threads: identity rows outside the row, a of its
            // first and c of its last equation 0, elements past the copied ones
            const int have = copied(row0) - sh;
#pragma unroll
            for (int e = 0; e < P; ++e) {
                const int i = i0 + e;
                const bool in = i >= 0 && i < nrow;
                if (in && i >= have) {
                    a[e] = ga[row0 + i];
                    b[e] = gb[row0 + i];
                    c[e] = gc[row0 + i];
                    d[e] = gd[row0 + i];
                }
                a[e] = in && i > 0 ? a[e] : 0.f;
                b[e] = in ? b[e] : 1.f;
                c[e] = in && i < nrow - 1 ? c[e] : 0.f;
                d[e] = in ? d[e] : 0.f;
            }
        }
        wm::wm_solve_inreg<P, 2, 1, true, PER_WARP>(a, b, c, d, log_tps, buf, tps, t, t, slots);
        float *xo = x + row0 + i0;
#pragma unroll
        for (int q = 0; q < P; q += 4) {
            const int i = i0 + q;
            if (i >= 0 && i + 3 < nrow) {
                __stcs(reinterpret_cast<float4 *>(xo + q), make_float4(d[q], d[q + 1], d[q + 2], d[q + 3]));
            } else {
#pragma unroll
                for (int e = q; e < q + 4; ++e)
                    if (i0 + e >= 0 && i0 + e < nrow) xo[e] = d[e];
            }
        }
    }
}

template <int P, int R, bool RAGGED>
const void *wm_func_r(int shuffle) {
    constexpr int MAXT = P >= 8 || R >= 8 ? 512 : 1024;
    return shuffle ? reinterpret_cast<const void *>(&tridiag_wm_kernel<P, R, 1, MAXT, RAGGED>)
                   : reinterpret_cast<const void *>(&tridiag_wm_kernel<P, R, 0, MAXT, RAGGED>);
}

template <int P, bool RAGGED>
const void *wm_func_p(int radix, int shuffle) {
    switch (radix) {
        case 2: return wm_func_r<P, 2, RAGGED>(shuffle);
        case 4: return wm_func_r<P, 4, RAGGED>(shuffle);
        case 8: return wm_func_r<P, 8, RAGGED>(shuffle);
        default: return nullptr;
    }
}

template <bool RAGGED>
const void *wm_func(int P, int radix, int shuffle) {
    switch (P) {
        case 2: return wm_func_p<2, RAGGED>(radix, shuffle);
        case 4: return wm_func_p<4, RAGGED>(radix, shuffle);
        case 8: return wm_func_p<8, RAGGED>(radix, shuffle);
        case 16: return wm_func_p<16, RAGGED>(radix, shuffle);
        default: return nullptr;
    }
}

}  // namespace

int tridiag_wm_smem_bytes(const bplg_plan &p, int64_t n) {
    const int64_t tps = n / p.P;
    return wm_warp_only(p.shuffle, tps) ? 0 : 4 * 16 * p.L;
}

bool tridiag_wm_launch_info(const bplg_plan &p, int64_t n, int64_t batch, Launch *out) {
    if (!plan_structurally_valid(p, BPLG_F32, n, nullptr)) return false;
    const void *f = wm_func<false>(p.P, p.radix, p.shuffle);
    if (!f) return false;
    out->func = f;
    out->threads = p.L;
    out->smem = tridiag_wm_smem_bytes(p, n);
    out->blocks = (batch + p.spb - 1) / p.spb;
    return true;
}

// Read (and optionally clear) the device error word of this file's kernels.
int tridiag_wm_device_status(int *flag, bool reset) {
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_device_error, sizeof(int));
    if (e != cudaSuccess) return cuda_error(e, "device status");
    if (reset && v) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_device_error, &zero, sizeof(int));
        if (e != cudaSuccess) return cuda_error(e, "device status reset");
    }
    *flag = v;
    return BPLG_OK;
}

// Which calls take it: lengths above 256 whose padded form wastes threads or has
// rows off 16-byte boundaries, unless
//   - a multiple of 4 above three quarters of the power of two, up to 2048, other than
//     1684 .. 1920 (five nearly full warps of P = 12): of the padded form's threads (P =
//     8) nearly all are busy, and without a slot in shared memory more of its blocks fit
//     an SM (2^24 unknowns, cost model's plan padded / bulk copies: n = 392 59 / 64 us,
//     500 52 / 55, 800 63 / 70, 1544 63 / 66, 2000 57 / 60, but 380 60 / 59, 764 65 / 60,
//     1532 63 / 56, 1800 60 / 58, 4032 72 / 69); up to 256 a block here is one warp with
//     half of its lanes idle;
//   - few systems, which take as long as one, the longer the more equations a thread
//     has (device time, padded / bulk copies: 76 systems of n = 300 2.5 / 3.1 us, 491 2.7
//     / 3.6, 1100 3.2 / 3.6, 3600 4.7 / 5.4, but 1025 4.4 / 3.6, 6500 6.8 / 6.5; the two
//     meet at 1800 systems of 300, 900 of 600, 350 of 1100, 450 of 1500, 300 of 2200 and
//     641, 150 of 901).
bool tridiag_wm_tma_applies(int64_t n, int64_t batch) {
    if (is_pow2(n) || n <= 256 || n > (int64_t(1) << kTridiagMaxLog)) return false;
    const bool aligned = n % 4 == 0;
    const int64_t few = aligned ? (n <= 384 ? 1824 : (n <= 1024 ? 608 : (n <= 2048 ? 304 : (n <= 4096 ? 152 : 0))))
                                : (n <= 640 ? 304 : (n <= 900 ? 152 : 0));
    const bool full = aligned && n < 2048 && 4 * n > 3 * next_pow2(n) && (n <= 1680 || n > 1920);
    return batch > few && !full;
}

// The padded kernel's plan for those calls above 256 whose power of two is at most 1024,
// without a plan tuned for it: P = 16, one system a block.  (The cost model's plan, P
// = 8, suits whole systems: n = 400 59.8 us at 2^24 unknowns, this one 53.8; 800 63.9,
// 55.6; and its sums, of twice the threads, are further from float64, 6.66e-8 against
// 6.41e-8.)
bool tridiag_wm_padded_plan(int64_t n, int64_t batch, bplg_plan *p) {
    const int64_t np = next_pow2(n);
    if (np == n || np < 512 || np > 1024 || cache_lookup(BPLG_OP_TRIDIAG_WM, BPLG_F32, np, batch, p)) return false;
    *p = {};
    p->op = BPLG_OP_TRIDIAG_WM;
    p->P = 16;
    p->spb = 1;
    p->radix = 2;
    p->shuffle = 1;
    plan_finalize(p, BPLG_F32, np);
    return true;
}

int tridiag_wm_tma_launch(const float *a, const float *b, const float *c, const float *d, float *x, int64_t n,
                          int64_t batch, cudaStream_t s) {
    const int max_shift = n % 4 == 0 ? 0 : (n % 2 == 0 ? 2 : 3);  // elements before a row in its first 16 bytes
    const auto threads = [&](int P) { return static_cast<int>((n + max_shift + 32 * P - 1) / (32 * P) * 32); };
    // P = 12, or 20 where that leaves fewer threads idle: one warp instead of two
    // (n = 385 .. 640), and above 2048 (n = 2500 0.0665 -> 0.0613 ms, 3500 0.0734 -> 0.0643,
    // but 3000 0.0600 against 0.0645 and 4500 0.0683 against 0.0698, whose rows fill
    // P = 12 better).  More than 448 threads of P = 12 leave one block per SM
    // (n = 5500 0.0866 ms against 0.0709 with P = 20).
    const int t12 = threads(12), t20 = threads(20);
    const bool p20 = t20 == 32 ? t12 > 32 : t12 > 448 || (n > 2048 && 20 * t20 * 100 <= 12 * t12 * 101);
    const int P = p20 ? 20 : 12, tps = p20 ? t20 : t12;
    const bool per_warp = tps > 288 || (p20 && tps > 32);
    const void *f = p20 ? (tps == 32    ? reinterpret_cast<const void *>(&tridiag_wm_tma_kernel<20, 32, 14, false>)
                           : tps <= 288 ? reinterpret_cast<const void *>(&tridiag_wm_tma_kernel<20, 288, 2, true>)
                                        : reinterpret_cast<const void *>(&tridiag_wm_tma_kernel<20, 416, 1, true>))
                        : (tps <= 288 ? reinterpret_cast<const void *>(&tridiag_wm_tma_kernel<12, 288, 3, false>)
                                      : reinterpret_cast<const void *>(&tridiag_wm_tma_kernel<12, 448, 2, true>));
    int log_tps = ilog2(next_pow2(tps)), nrow = static_cast<int>(n);
    const int smem = 4 * 16 * ((1 << log_tps) >> (per_warp ? 5 : 0)) + 4 * 4 * tps * P;
    int rc = check_grid(batch, "tridiag (Wang-Mou)");  // one block a system at most, as the padded kernel
    if (rc == BPLG_OK) rc = ensure_smem_attr(f, smem);
    if (rc != BPLG_OK) return rc;
    int64_t grid = 0;
    rc = persistent_grid(f, tps, smem, batch, &grid);
    if (rc != BPLG_OK) return rc;
    void *args[] = {(void *)&a, (void *)&b, (void *)&c, (void *)&d, (void *)&x, &log_tps, &batch, &nrow};
    cudaError_t e = cudaLaunchKernel(f, dim3(static_cast<unsigned>(grid)), dim3(tps), args, static_cast<size_t>(smem), s);
    return e == cudaSuccess ? BPLG_OK : launch_error(e, "tridiag (Wang-Mou, bulk-copy) launch", f, grid, tps, smem);
}

int tridiag_wm_launch(const bplg_plan &p, const float *a, const float *b, const float *c, const float *d, float *x,
                      int64_t n, int64_t batch, cudaStream_t s) {
    // a plan made for the next power of two runs a length-n system padded
    const int64_t np = p.n > 0 ? p.n : n;
    if (np < n || (np != n && np / 2 >= n)) return set_error(BPLG_ERR_INVALID_PLAN, "tridiag (Wang-Mou): plan is for another n");
    Launch li;
    if (!tridiag_wm_launch_info(p, np, batch, &li))
        return set_error(BPLG_ERR_INVALID_PLAN, "tridiag (Wang-Mou): plan has no kernel");
    if (np != n) li.func = wm_func<true>(p.P, p.radix, p.shuffle);
    int rc = check_grid(li.blocks, "tridiag (Wang-Mou)");
    if (rc != BPLG_OK) return rc;
    rc = ensure_smem_attr(li.func, li.smem);
    if (rc != BPLG_OK) return rc;
    int logn = ilog2(np), log_tps = ilog2(np / p.P), spb = p.spb, nrow = static_cast<int>(n);
    void *args[] = {(void *)&a, (void *)&b, (void *)&c, (void *)&d, (void *)&x, &logn, &log_tps, &spb, &batch, &nrow};
    cudaError_t e = cudaLaunchKernel(li.func, dim3(static_cast<unsigned>(li.blocks)), dim3(li.threads), args,
                                     static_cast<size_t>(li.smem), s);
    return e == cudaSuccess ? BPLG_OK
                            : launch_error(e, "tridiag (Wang-Mou) launch", li.func, li.blocks, li.threads, li.smem);
}

}  // namespace bplg
