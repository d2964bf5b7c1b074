// The FFT of lengths with prime factors 7 to 31: see fft_prime.cuh.
//
// A block holds spb signals.  Its threads take the spb n / r butterflies of a
// stage in turn, signal-major, so that consecutive threads read consecutive
// elements (runs of m) and write consecutive ones; a butterfly's outputs go
// straight to the other of two shared-memory buffers (one barrier a stage), so a
// thread holds one butterfly's inputs only.  The first stage reads global memory
// and the last one writes it.
//
// A prime radix is summed from its definition in halves: with t_k = v_k + v_{R-k}
// and d_k = v_k - v_{R-k}, outputs q and R - q are b_q +- i u_q,
// b_q = v_0 + sum_k cos(2 pi q k / R) t_k, u_q = sum_k sin(2 pi q k / R) d_k:
// (R - 1)^2 fused multiply-adds for R points, 29 a point at R = 31.
// Such lengths went through Bluestein's identity before, two power-of-two
// transforms of up to 4 n points each.  Measured at 2^24 points, Bluestein (with
// its exchange-free product) -> this kernel: n = 77 0.148 -> 0.0495 ms, 1001 0.133 ->
// 0.061 (65 % of the copy bandwidth), 4004 0.23 -> 0.088; 2^22 points: 4199 0.267
// -> 0.027, 12012 0.237 -> 0.050.  Error against float64 at n = 1001: 1.8e-7 ->
// 1.1e-7.  It is bound by the L1 data pipe up to radix 13 and by occupancy (128
// registers) for the largest primes; one prime alone (n = 31, 0.099 ms) by its
// strided global accesses.
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "fft_mixed.cuh"
#include "fft_prime.cuh"
#include "internal.h"

namespace bplg {

namespace {

using mixed_detail::cos_2pi;
using mixed_detail::dft_any;
using mixed_detail::sin_2pi;

__device__ __forceinline__ uint32_t fast_div(uint32_t x, int d, uint32_t inv) { return d > 1 ? __umulhi(x, inv) : x; }

// cos and sin of 2 pi k / R, k < R, evaluated once at compile time in float64
template <int R>
struct PrimeRoots {
    float c[R] = {}, s[R] = {};
    constexpr PrimeRoots() {
        for (int k = 0; k < R; ++k) {
            c[k] = static_cast<float>(cos_2pi(k, R));
            s[k] = static_cast<float>(sin_2pi(k, R));
        }
    }
};

// v -> store(q, y_q), R an odd prime
template <int R, int DIR, class Store>
__device__ __forceinline__ void dft_prime(float2 (&v)[R], Store store) {
    constexpr int H = (R - 1) / 2;
    constexpr PrimeRoots<R> W;
    float2 y0 = v[0];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        const float2 t = cadd(v[k], v[R - k]), d = csub(v[k], v[R - k]);
        v[k] = t;
        v[R - k] = d;
        y0 = cadd(y0, t);
    }
    store(0, y0);
#pragma unroll
    for (int q = 1; q <= H; ++q) {
        float2 b = v[0], u = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            const float c = W.c[q * k % R], s = DIR * W.s[q * k % R];
            b.x = fmaf(c, v[k].x, b.x);
            b.y = fmaf(c, v[k].y, b.y);
            u.x = k == 1 ? s * v[R - k].x : fmaf(s, v[R - k].x, u.x);
            u.y = k == 1 ? s * v[R - k].y : fmaf(s, v[R - k].y, u.y);
        }
        store(q, make_float2(b.x - u.y, b.y + u.x));  // b + i u
        store(R - q, make_float2(b.x + u.y, b.y - u.x));
    }
}

// One stage of radix R over the block's `live` signals.
template <int R, int DIR, bool FIRST, bool LAST>
__device__ __forceinline__ void prime_stage(const PrimePlan &p, int s, const float2 *src, float2 *dst,
                                            const float2 *__restrict__ tw, int live) {
    const int n = p.n, nb = n / R, m = LAST ? 1 : p.m[s], L = FIRST ? 1 : p.L[s], lm = L * m;
    const float2 *tws = tw + (L - p.r[0]);  // this stage's block of the table
    for (uint32_t i = threadIdx.x; i < static_cast<uint32_t>(live * nb); i += blockDim.x) {
        const uint32_t sg = fast_div(i, nb, p.inv_nb[s]);
        const int b = static_cast<int>(i - sg * nb);
        const int j = FIRST ? 0 : (LAST ? b : static_cast<int>(fast_div(b, m, p.inv_m[s])));
        const float2 *in = src + sg * n + b + (R - 1) * j * m;
        float2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = FIRST ? __ldcs(in + q * m) : in[q * m];
        if constexpr (!FIRST) {
#pragma unroll
            for (int q = 1; q < R; ++q) {
                float2 w = __ldg(tws + (q - 1) * L + j);
                if (DIR > 0) w.y = -w.y;
                v[q] = cmul(v[q], w);
            }
        }
        float2 *o = dst + sg * n + b;
        auto store = [&](int q, float2 y) {
            if constexpr (LAST)
                __stcs(o + q * lm, y);
            else
                o[q * lm] = y;
        };
        if constexpr (R >= 7 && R % 2 == 1 && R != 9) {
            dft_prime<R, DIR>(v, store);
        } else {
            dft_any<R, DIR>(v);
#pragma unroll
            for (int q = 0; q < R; ++q) store(q, v[q]);
        }
    }
}

// MAXR: the largest prime of the lengths this kernel serves (13, 19 or 31)
template <int MAXR, int DIR, bool FIRST, bool LAST>
__device__ __forceinline__ void prime_dispatch(const PrimePlan &p, int s, const float2 *src, float2 *dst,
                                               const float2 *__restrict__ tw, int live) {
#define BPLG_STAGE(R) \
    case R: prime_stage<R, DIR, FIRST, LAST>(p, s, src, dst, tw, live); break;
    switch (p.r[s]) {
        BPLG_STAGE(7)
        BPLG_STAGE(11)
        BPLG_STAGE(13)
        default:
            if constexpr (MAXR >= 19) {
                switch (p.r[s]) {
                    BPLG_STAGE(17)
                    BPLG_STAGE(19)
                    default: break;
                }
            }
            if constexpr (MAXR >= 31) {
                switch (p.r[s]) {
                    BPLG_STAGE(23)
                    BPLG_STAGE(29)
                    BPLG_STAGE(31)
                    default: break;
                }
            }
            if constexpr (!FIRST) {  // the first stage is the largest prime
                switch (p.r[s]) {
                    BPLG_STAGE(2)
                    BPLG_STAGE(3)
                    BPLG_STAGE(4)
                    BPLG_STAGE(5)
                    BPLG_STAGE(6)
                    BPLG_STAGE(8)
                    BPLG_STAGE(9)
                    BPLG_STAGE(10)
                    default: break;
                }
            }
    }
#undef BPLG_STAGE
}

template <int MAXR, int DIR>
__global__ void __launch_bounds__(kPrimeMaxThreads, MAXR == 13 ? 4 : (MAXR == 19 ? 3 : 2))
    fft_prime_kernel(const float2 *in, float2 *out, const float2 *__restrict__ tw, const __grid_constant__ PrimePlan p,
                     int64_t batch) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *buf = reinterpret_cast<float2 *>(smem_raw);
    const int64_t sig0 = static_cast<int64_t>(blockIdx.x) * p.spb;
    const int live = batch - sig0 < p.spb ? static_cast<int>(batch - sig0) : p.spb;
    const float2 *g = in + sig0 * p.n;
    float2 *o = out + sig0 * p.n;
    if (p.stages == 1) {
        prime_dispatch<MAXR, DIR, true, true>(p, 0, g, o, tw, live);
        return;
    }
    const int size = p.spb * p.n;
    prime_dispatch<MAXR, DIR, true, false>(p, 0, g, buf, tw, live);
    __syncthreads();
    for (int s = 1; s < p.stages - 1; ++s) {
        prime_dispatch<MAXR, DIR, false, false>(p, s, buf + ((s - 1) & 1) * size, buf + (s & 1) * size, tw, live);
        __syncthreads();
    }
    prime_dispatch<MAXR, DIR, false, true>(p, p.stages - 1, buf + ((p.stages - 2) & 1) * size, o, tw, live);
}

std::mutex g_mu;
struct Entry {
    PrimePlan plan;
    float2 *tw;  // the stage twiddles
};
std::map<std::pair<int, int64_t>, Entry> g_entries;  // (device, n)

// stage s >= 1: W_n^(q j m), q = 1 .. r - 1, j < L, at [L - r_0 + (q - 1) L + j]
int entry_for(int64_t n, Entry *out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_entries.find(std::make_pair(dev, n));
    if (it != g_entries.end()) {
        *out = it->second;
        return BPLG_OK;
    }
    const PrimePlan p = prime_plan(n);
    if (p.stages == 0) return set_error(BPLG_ERR_UNSUPPORTED_SIZE, "fft (prime radices): unsupported length");
    std::vector<float2> h;
    h.reserve(static_cast<size_t>(p.n));
    for (int s = 1; s < p.stages; ++s)
        for (int q = 1; q < p.r[s]; ++q)
            for (int j = 0; j < p.L[s]; ++j) {
                const double ang = -2.0 * M_PI * static_cast<double>(int64_t(q) * j * p.m[s]) / static_cast<double>(p.n);
                h.push_back(make_float2(static_cast<float>(std::cos(ang)), static_cast<float>(std::sin(ang))));
            }
    if (h.empty()) h.push_back(make_float2(1.f, 0.f));  // one stage: no twiddles
    float2 *d = nullptr;
    if ((e = cudaMalloc(&d, h.size() * sizeof(float2))) != cudaSuccess) return cuda_error(e, "prime-radix twiddles");
    const int rc = upload(d, h.data(), h.size() * sizeof(float2), "prime-radix twiddles upload");
    if (rc != BPLG_OK) {
        cudaFree(d);
        return rc;
    }
    *out = g_entries[std::make_pair(dev, n)] = Entry{p, d};
    return BPLG_OK;
}

}  // namespace

bool fft_prime_applies(int64_t n) {
    if (n < 7 || n > kPrimeMaxLen) return false;
    bool large = false;
    for (int q : {2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31})
        while (n % q == 0) {
            n /= q;
            large = large || q >= 7;
        }
    return n == 1 && large;
}

template <int DIR>
static const void *prime_func(int tier) {
    return tier == 13   ? reinterpret_cast<const void *>(&fft_prime_kernel<13, DIR>)
           : tier == 19 ? reinterpret_cast<const void *>(&fft_prime_kernel<19, DIR>)
                        : reinterpret_cast<const void *>(&fft_prime_kernel<31, DIR>);
}

int fft_prime_launch(const void *in, void *out, int64_t n, int64_t batch, int dir, cudaStream_t s) {
    Entry en;
    int rc = entry_for(n, &en);
    if (rc != BPLG_OK) return rc;
    const PrimePlan &p = en.plan;
    const float2 *tw = en.tw;
    const int tier = prime_tier(p.r[0]);
    const void *f = dir < 0 ? prime_func<-1>(tier) : prime_func<1>(tier);
    const int smem = prime_smem(p);
    rc = ensure_smem_attr(f, smem);
    if (rc != BPLG_OK) return rc;
    const int64_t blocks = (batch + p.spb - 1) / p.spb;
    rc = check_grid(blocks, "fft (prime radices)");
    if (rc != BPLG_OK) return rc;
    const float2 *xi = static_cast<const float2 *>(in);
    float2 *xo = static_cast<float2 *>(out);
    void *args[] = {(void *)&xi, (void *)&xo, (void *)&tw, (void *)&p, &batch};
    cudaError_t e = cudaLaunchKernel(f, dim3(static_cast<unsigned>(blocks)), dim3(p.threads), args,
                                     static_cast<size_t>(smem), s);
    return e == cudaSuccess ? BPLG_OK : launch_error(e, "fft (prime radices) launch", f, blocks, p.threads, smem);
}

}  // namespace bplg
