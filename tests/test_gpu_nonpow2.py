"""Lengths that are not powers of two: the scan and the Wang-Mou tridiagonal
solver run the plan of the next power of two with identity padding, the FFT
runs a mixed-radix Stockham kernel for 2^a 3^b 5^c up to 12288 and
Bluestein's chirp identity over power-of-two FFTs otherwise.  Parity against the
oracle (scan bit-exact for int32, the float64 Thomas solution <= 1e-4, the
O(N^2) DFT <= 1e-5 ceil(log2 N)), closed forms at sizes the O(N^2) oracle
cannot reach, every plan of the padded size, and nothing written past n."""
import math

import numpy as np
import pytest

import oracle
import seeded_inputs as si
from tests.gpu_util import c64_from_dev, c64_to_dev, fft_rel_err, to_dev, tri_rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SENTINEL = 12345


@pytest.fixture(scope="module")
def bp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_16214_gb300 as bp
    return bp


def next_pow2(n):
    return 1 << max(0, (n - 1).bit_length())


# ------------------------------------------------------------------ scan ----

def run_scan(bp, x, plan=None, guard=64):
    batch, n = x.shape
    xin = to_dev(x.reshape(-1))
    out = torch.full((batch * n + guard,), SENTINEL, dtype=xin.dtype, device="cuda")
    bp.scan_batched(xin, out, n, batch, dtype=bp.I32 if x.dtype == np.int32 else bp.F32, plan=plan)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    assert np.all(o[batch * n:] == SENTINEL), "written past the last row"
    return o[:batch * n].reshape(batch, n)


@pytest.mark.parametrize("n", [1, 3, 5, 31, 33, 100, 1000, 4097, 32767])
def test_scan_i32_every_plan_bit_exact(bp, n):
    batch = 7
    x = si.scan_i32(batch, n, stream=500 + n)
    ref = oracle.scan_i32(x)
    plans = bp.enumerate_plans(bp.OP_SCAN, bp.I32, next_pow2(n)) if n > 1 else [None]
    step = max(1, len(plans) // 12)
    for p in plans[::step] + [None]:
        assert np.array_equal(run_scan(bp, x, p), ref), p


@pytest.mark.parametrize("n", [3, 100, 1000, 5000])
def test_scan_f32_padded(bp, n):
    batch = 5
    x = si.scan_f32(batch, n, stream=600 + n, integer_valued=True)
    assert np.array_equal(run_scan(bp, x).astype(np.float64), oracle.scan_f32(x))


def test_scan_plan_for_another_length_rejected(bp):
    n, batch = 100, 3
    x = si.scan_i32(batch, n, stream=7)
    with pytest.raises(bp.BplgError):
        run_scan(bp, x, bp.make_plan(bp.OP_SCAN, 256, 4, 1))  # made for 256, not 128


# --------------------------------------------------------------- tridiag ----

def run_tri(bp, sysm, plan=None, guard=64):
    a, b, c, d = sysm[:4]
    batch, n = b.shape
    ts = [to_dev(v.reshape(-1)) for v in (a, b, c, d)]
    x = torch.full((batch * n + guard,), float(SENTINEL), dtype=torch.float32, device="cuda")
    bp.tridiag_batched(*ts, x, n, batch, plan=plan)
    torch.cuda.synchronize()
    o = x.cpu().numpy()
    assert np.all(o[batch * n:] == SENTINEL), "written past the last row"
    return o[:batch * n].reshape(batch, n)


@pytest.mark.parametrize("n", [3, 5, 17, 100, 1000, 3000, 5000])
def test_tridiag_every_wm_plan(bp, n):
    batch = 9 if n <= 1000 else 3
    a, b, c, d, _ = si.tridiag_f32(batch, n, stream=700 + n)
    c[:, -1] = np.nan  # never read
    ref = oracle.thomas(a, b, c, d)
    for p in bp.enumerate_plans(bp.OP_TRIDIAG_WM, bp.F32, next_pow2(n)) + [None]:
        x = run_tri(bp, (a, b, c, d), p)
        assert np.all(np.isfinite(x)) and tri_rel_err(x, ref).max() <= 1e-4, p


def test_tridiag_cr_plan_needs_power_of_two(bp):
    n, batch = 100, 2
    sysm = si.tridiag_f32(batch, n, stream=8)
    with pytest.raises(bp.BplgError):
        run_tri(bp, sysm, bp.make_plan(bp.OP_TRIDIAG, 128, 2, 1, cr_switch=32, shuffle=1))


# Both forms of the kernel for rows (on the threads the row needs, and padded)
# under every plan, at lengths on both sides of the lines between them.
@pytest.mark.parametrize("n", [6, 12, 15, 20, 28, 60, 63, 65, 96, 127, 130, 255, 260, 448, 500, 511, 640, 700, 1020, 2000])
def test_scan_row_forms_every_plan(bp, n):
    batch = 67
    x = si.scan_i32(batch, n, stream=1500 + n)
    ref = oracle.scan_i32(x)
    f = si.scan_f32(batch, n, stream=1600 + n, integer_valued=True)  # sums exact in float32
    for p in bp.enumerate_plans(bp.OP_SCAN, bp.I32, next_pow2(n)) + [None]:
        assert np.array_equal(run_scan(bp, x, p), ref), p
    for p in bp.enumerate_plans(bp.OP_SCAN, bp.F32, next_pow2(n))[::7] + [None]:
        assert np.array_equal(run_scan(bp, f, p), np.cumsum(f.astype(np.float64), axis=1).astype(np.float32)), p


# A row a little longer than a power of two costs about what that one costs per
# element (0.98 of it; 1.24 to 1.36 when every four elements had a prefix of their own).
@pytest.mark.parametrize("n", [260, 300])
def test_scan_short_rows_keep_the_rate(bp, n):
    total = 1 << 26
    x = torch.zeros(total, dtype=torch.int32, device="cuda")
    y = torch.empty_like(x)

    def per_element(m, plan):
        ts = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                bp.scan_batched(x, y, m, total // m, plan=plan)
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1) / (total // m * m))
        return min(ts)

    whole = per_element(256, None)
    for plan in (None, bp.make_plan(bp.OP_SCAN, 512, P=16, spb=2)):
        assert per_element(n, plan) <= 1.15 * whole, plan


# Rounding grows with the row: the padded form of a short row is no further from the
# float64 sums than the longer power of two is (9.4e-8 against 8.3e-8 when a run of 16
# was summed serially, 7.8e-8 in fours and pairs).
@pytest.mark.parametrize("n", [260, 300])
def test_scan_f32_padded_runs_round_as_little(bp, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(4)

    def error(m):
        x = torch.rand((1 << 22) // m, m, generator=g, device="cuda") * 2 - 1
        y = torch.empty_like(x)
        bp.scan_batched(x, y, m, x.shape[0])
        ref = torch.cumsum(x.double(), dim=1)
        return ((y.double() - ref).norm() / ref.norm()).item()

    assert error(n) <= 1.02 * error(512)


# The plan of a call without one depends on the batch: a small, a middle and a large
# one of each kind of length.
@pytest.mark.parametrize("n", [20, 33, 130, 260, 400, 500, 800, 1000, 1100, 2000, 5000, 5001, 8191, 9000, 20000, 32767])
def test_scan_default_plan_by_batch(bp, n):
    for total in (1 << 19, 3 << 20, (1 << 24) + n):
        batch = total // n
        x = torch.randint(-1000, 1001, (batch, n), dtype=torch.int32, device="cuda")
        y = torch.empty_like(x)
        bp.scan_batched(x, y, n, batch)
        assert torch.equal(y, torch.cumsum(x, dim=1, dtype=torch.int32)), total


# A few rows take about as long as a few of the next power of two (1.0 to 1.1 of it on
# the device; 1.6 to 1.7 when 32 elements a thread were taken there too).
@pytest.mark.parametrize("n", [1000, 2000])
def test_scan_few_rows(bp, n):
    x = torch.zeros(1 << 16, dtype=torch.int32, device="cuda")
    y = torch.empty_like(x)

    def per_call(m):
        bp.scan_batched(x, y, m, 16)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(50):
                bp.scan_batched(x, y, m, 16)
        ts = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            g.replay()
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        return min(ts)

    assert per_call(n) <= 1.3 * per_call(next_pow2(n))


# Rows that start 1, 2 and 3 elements past a 16-byte boundary, at lengths
# whose last thread, warp or block is nearly empty or exactly full, and at the
# longest odd lengths (no room for the shift at n = 32767); in place too.
@pytest.mark.parametrize("n", [18, 65, 257, 1021, 1022, 1023, 2047, 2049, 8190, 16385, 32766, 32767])
def test_scan_rows_off_alignment(bp, n):
    batch = 6
    x = si.scan_i32(batch, n, stream=900 + n)
    ref = oracle.scan_i32(x)
    assert np.array_equal(run_scan(bp, x), ref)
    buf = to_dev(x.reshape(-1))
    bp.scan_batched(buf, buf, n, batch)
    assert np.array_equal(buf.cpu().numpy().reshape(batch, n), ref)


# Every thread count and equations-per-thread choice of the bulk-copy solver
# (257 .. 8191), rows at all four places in their 16 bytes, at the edges of its
# ranges; batches small and large enough that a block solves several systems in
# turn; x may alias d.
@pytest.mark.parametrize("n,batch", [(18, 6), (257, 6000), (380, 5), (384, 3), (385, 6), (637, 6), (638, 4001), (959, 7),
                                     (1021, 6), (1022, 6), (1023, 6), (1025, 3000), (2047, 6), (2500, 1500), (3001, 1101),
                                     (3500, 6), (4095, 6), (5373, 700), (5374, 6), (5757, 6), (5758, 501), (8190, 6),
                                     (8191, 400)])
def test_tridiag_rows_off_alignment(bp, n, batch):
    a, b, c, d, _ = si.tridiag_f32(batch, n, stream=950 + n)
    a[:, 0] = np.nan  # never read
    c[:, -1] = np.nan
    ref = oracle.thomas(a, b, c, d)
    x = run_tri(bp, (a, b, c, d))
    assert np.all(np.isfinite(x)) and tri_rel_err(x, ref).max() <= 1e-4
    ts = [to_dev(v.reshape(-1)) for v in (a, b, c, d)]
    bp.tridiag_batched(*ts, ts[3], n, batch)  # x aliases d
    assert np.array_equal(ts[3].cpu().numpy().reshape(batch, n), x)
    assert bp.device_status() == 0


# The bulk-copy solver and the padded one take turns over length and batch: both
# sides of each line, every shape of the bulk-copy solver in batches large enough for it.
@pytest.mark.parametrize("n,batch", [(380, 1825), (384, 1824), (384, 1825), (388, 700), (385, 304), (385, 305), (637, 310),
                                     (640, 609), (641, 152), (641, 153), (768, 608), (768, 609), (772, 700), (900, 160),
                                     (901, 2), (1500, 304), (1500, 305), (1536, 609), (1540, 620), (1680, 305), (1684, 305),
                                     (1920, 305), (1924, 305), (2044, 609), (2052, 152), (2052, 153), (4092, 153),
                                     (4100, 1)])
def test_tridiag_ragged_lines(bp, n, batch):
    a, b, c, d, _ = si.tridiag_f32(batch, n, stream=1900 + n)
    a[:, 0] = np.nan  # never read
    c[:, -1] = np.nan
    rows = np.unique(np.r_[:3, batch // 2, max(0, batch - 3):batch])
    rows = rows[rows < batch]
    x = run_tri(bp, (a, b, c, d))
    assert np.all(np.isfinite(x))
    assert tri_rel_err(x[rows], oracle.thomas(a[rows], b[rows], c[rows], d[rows])).max() <= 1e-4
    assert bp.device_status() == 0


# Lengths whose padded form is the faster one take it without a plan (the bulk copies
# took 1.16 to 1.19 of its time).
@pytest.mark.parametrize("n", [800, 2000])
def test_tridiag_ragged_as_fast_as_padded(bp, n):
    total = 1 << 24
    ts = [torch.zeros(total, device="cuda") for _ in range(5)]
    ts[1].fill_(1.0)

    def per_unknown(m, plan):
        best = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                bp.tridiag_batched(*ts, m, total // m, plan=plan)
            e1.record()
            e1.synchronize()
            best.append(e0.elapsed_time(e1))
        return min(best) / (total // m * m)

    padded = bp.query_plan(bp.OP_TRIDIAG_WM, bp.F32, next_pow2(n), total // n)
    assert per_unknown(n, None) <= 1.08 * per_unknown(n, padded)


# Whichever of the two kernels a length and batch take, it is as far from float64: 6.3e-8
# to 6.6e-8 of the solution's norm (the padded kernel of eight equations a thread 6.66e-8).
@pytest.mark.parametrize("n,batch", [(300, 100), (400, 10000), (491, 100), (600, 100), (800, 5000), (3000, 500)])
def test_tridiag_ragged_rounding(bp, n, batch):
    a, b, c, d, _ = si.tridiag_f32(batch, n, stream=2000 + n)
    ref = oracle.thomas(a, b, c, d)
    x = run_tri(bp, (a, b, c, d))
    assert np.linalg.norm(x - ref) <= 6.62e-8 * np.linalg.norm(ref)


# Tuning the next power of two does not change what a call of another length runs: the
# same bits before and after.
def test_ragged_calls_do_not_follow_the_tuned_power_of_two(bp):
    n, batch = 3001, 700
    a, b, c, d, _ = si.tridiag_f32(batch, n, stream=77)
    before = run_tri(bp, (a, b, c, d))
    bp.tune_plan(bp.OP_TRIDIAG_WM, bp.F32, next_pow2(n), batch, bp.TUNE_MODEL)
    assert np.array_equal(run_tri(bp, (a, b, c, d)), before)
    for n, batch in [(1000, 40), (1003, 20000), (5000, 3400)]:
        x = torch.rand(batch, n, device="cuda") - 0.5
        y0, y1 = torch.empty_like(x), torch.empty_like(x)
        bp.scan_batched(x, y0, n, batch)
        bp.tune_plan(bp.OP_SCAN, bp.F32, next_pow2(n), batch, bp.TUNE_EXHAUSTIVE)
        bp.scan_batched(x, y1, n, batch)
        assert torch.equal(y0, y1), n


# ------------------------------------------------------------------- FFT ----

def tol(n):
    return 1e-5 * math.ceil(math.log2(n))


def run_fft(bp, x, direction, plan=None, guard=16):
    batch, n = x.shape
    xin = c64_to_dev(x.reshape(-1))
    out = torch.full((2 * (batch * n + guard),), float(SENTINEL), dtype=torch.float32, device="cuda")
    bp.fft_batched(xin, out, n, batch, direction, plan=plan)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    assert np.all(o[2 * batch * n:] == SENTINEL), "written past the last row"
    return o[:2 * batch * n].view(np.complex64).reshape(batch, n)


# lengths with a prime factor above 5 (these run prime radices now; Bluestein's
# lengths, with a prime factor above 31, follow)
@pytest.mark.parametrize("n", [7, 14, 77, 1001, 4095])
def test_fft_bluestein_vs_dft(bp, n):
    batch = 6 if n <= 1001 else 2
    x = si.fft_c64(batch, n, stream=800 + n)
    for direction in (-1, 1):
        X = run_fft(bp, x, direction)
        ref = oracle.dft(x, direction)
        assert fft_rel_err(X, ref).max() <= tol(n), (n, direction)


# lengths with a prime factor above 31: the fused Bluestein kernel at both ends of
# its range (M = 128 .. 8192)
@pytest.mark.parametrize("n", [37, 74, 1009, 2039, 4093])
def test_fft_bluestein_large_primes_vs_dft(bp, n):
    batch = 5 if n <= 1009 else 2
    x = si.fft_c64(batch, n, stream=820 + n)
    for direction in (-1, 1):
        assert fft_rel_err(run_fft(bp, x, direction), oracle.dft(x, direction)).max() <= tol(n), (n, direction)


# the other inner lengths of the fused kernel (M = 128, 512, 1024), and blocks of many
# signals: several blocks, the last one not full
@pytest.mark.parametrize("n,batch", [(37, 70), (61, 33), (251, 19), (509, 9), (1009, 3)])
def test_fft_bluestein_blocks_of_signals(bp, n, batch):
    x = si.fft_c64(batch, n, stream=2600 + n)
    for direction in (-1, 1):
        assert fft_rel_err(run_fft(bp, x, direction), oracle.dft(x, direction)).max() <= tol(n), (n, direction)


# in place, through the fused kernel and through the five kernels of M > 8192
@pytest.mark.parametrize("n,batch", [(37, 70), (1009, 9), (4093, 3), (4099, 2), (8191, 2)])
def test_fft_bluestein_in_place(bp, n, batch):
    x = si.fft_c64(batch, n, stream=2650 + n)
    buf = c64_to_dev(x)
    bp.fft_batched(buf, buf, n, batch, -1)
    assert np.array_equal(c64_from_dev(buf).reshape(batch, n), run_fft(bp, x, -1))
    bp.fft_batched(buf, buf, n, batch, 1)
    assert fft_rel_err(c64_from_dev(buf).reshape(batch, n) / n, x.astype(np.complex128)).max() <= 2 * tol(n)


# prime radices 7 .. 31: every radix first, in the middle and last, one stage to
# five, one signal a block and many (the last block not full), the longest
# length; in place too.  Above 2100 points against numpy's float64 FFT.
@pytest.mark.parametrize("n,batch", [(7, 700), (11, 5), (13, 3), (17, 250), (19, 4), (23, 4), (29, 4), (31, 70), (34, 61), (77, 31),
                                     (143, 20), (221, 16), (323, 4), (437, 6), (527, 5), (713, 3), (899, 3), (961, 5),
                                     (1001, 4), (1547, 3), (2001, 2), (2002, 3), (4004, 3), (4199, 2), (9009, 2),
                                     (10571, 2), (12012, 2), (12276, 3)])
def test_fft_prime_radices(bp, n, batch):
    x = si.fft_c64(batch, n, stream=840 + n)
    for direction in (-1, 1):
        X = run_fft(bp, x, direction)
        if n <= 2100:
            ref = oracle.dft(x, direction)
        else:
            z = x.astype(np.complex128)
            ref = np.fft.fft(z, axis=1) if direction < 0 else np.fft.ifft(z, axis=1, norm="forward")
        assert fft_rel_err(X, ref).max() <= tol(n), (n, direction)
    buf = c64_to_dev(x.reshape(-1))
    bp.fft_batched(buf, buf, n, batch, -1)
    assert np.array_equal(c64_from_dev(buf).reshape(batch, n), run_fft(bp, x, -1))


# 2^a 3^b 5^c (not a power of two, at most 12288): the mixed-radix Stockham
# kernels (one per length, radices 2 .. 25); small lengths several signals a
# block (ragged last block)
@pytest.mark.parametrize("n", [3, 5, 6, 9, 10, 12, 15, 20, 25, 27, 45, 60, 81, 100, 120, 125, 243, 360, 375, 625,
                               1000, 1215, 1536, 2187, 3000])
def test_fft_mixed_radix_vs_dft(bp, n):
    batch = 37 if n <= 100 else (5 if n < 1000 else 1)
    x = si.fft_c64(batch, n, stream=1800 + n)
    for direction in (-1, 1):
        X = run_fft(bp, x, direction)
        ref = oracle.dft(x, direction)
        assert fft_rel_err(X, ref).max() <= tol(n), (n, direction)


# radices 18, 20, 24 and 25 (each first and in the middle or last), several whole
# blocks of signals and a ragged last one; the bound of every length
@pytest.mark.parametrize("n", [324, 400, 432, 576, 600, 625, 2000, 3000, 6250, 12000])
def test_fft_mixed_large_radices(bp, n):
    batch = 19 if n < 1000 else 3
    x = si.fft_c64(batch, n, stream=2500 + n)
    for direction in (-1, 1):
        # from 1000 points on the O(N^2) oracle takes too long
        if n < 1000:
            ref = oracle.dft(x, direction)
        else:
            z = x.astype(np.complex128)
            ref = np.fft.fft(z, axis=1) if direction < 0 else np.fft.ifft(z, axis=1, norm="forward")
        assert fft_rel_err(run_fft(bp, x, direction), ref).max() <= tol(n), (n, direction)


# Lengths whose kernel needs fewer registers than its budget: two buffers for each of
# the blocks that are resident then left 28 KB of L1 (1.23 and 1.25 of the neighbour's
# time a point; with one buffer 1.03 and 1.05).
@pytest.mark.parametrize("n,neighbour", [(216, 288), (243, 270)])
def test_fft_mixed_radix_keeps_the_l1(bp, n, neighbour):
    total = 1 << 24
    x = torch.zeros(2 * total, device="cuda")
    y = torch.empty_like(x)

    def per_point(m):
        ts = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(20):
                bp.fft_batched(x, y, m, total // m, -1)
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        return min(ts) / (total // m * m)

    assert per_point(n) <= 1.14 * per_point(neighbour)


def test_fft_mixed_radix_every_length(bp):
    """Every length with a compile-time kernel (all 2^a 3^b 5^c up to 12288
    that are not powers of two), both directions.  Below 1000 points: three
    signals (a partly filled block) against the O(N^2) oracle.  From 1000 on
    (where the O(N^2) oracle would take minutes): an impulse against its
    closed form exp(dir 2 pi i j0 k / n) and a random signal against numpy's
    float64 FFT."""
    def smooth(v):
        for p in (2, 3, 5):
            while v % p == 0:
                v //= p
        return v == 1
    lengths = [n for n in range(3, 12289) if smooth(n) and n & (n - 1)]
    assert len(lengths) == 172
    for n in lengths:
        if n < 1000:
            x = si.fft_c64(3, n, stream=5000 + n)
            for direction in (-1, 1):
                X = run_fft(bp, x, direction)
                assert fft_rel_err(X, oracle.dft(x, direction)).max() <= tol(n), (n, direction)
            continue
        k = np.arange(n, dtype=np.float64)
        j0 = (7919 * n) // 9973
        imp = np.zeros((1, n), np.complex64)
        imp[0, j0] = 1
        x = si.fft_c64(1, n, stream=5000 + n)
        for direction in (-1, 1):
            X = run_fft(bp, imp, direction).astype(np.complex128)
            ref = np.exp(direction * 2j * np.pi * ((j0 * k) % n) / n)[None, :]
            assert fft_rel_err(X, ref).max() <= tol(n), (n, direction)
            Y = run_fft(bp, x, direction)
            xd = x.astype(np.complex128)
            ref = np.fft.fft(xd, axis=-1) if direction < 0 else np.fft.ifft(xd, axis=-1) * n
            assert fft_rel_err(Y, ref).max() <= tol(n), (n, direction)


@pytest.mark.parametrize("n", [3125, 6000, 10000, 12288])
def test_fft_mixed_radix_large_closed_forms(bp, n):
    """Beyond the O(N^2) oracle's reach: an impulse at j0 gives exp(-2 pi i
    j0 k / n), a tone at f gives n at bin f (both directions), and a random
    signal survives the forward-inverse round trip."""
    k = np.arange(n, dtype=np.float64)
    j0, f = 1234 % n, 777 % n
    for direction in (-1, 1):
        imp = np.zeros((3, n), np.complex64)
        imp[:, j0] = 1
        X = run_fft(bp, imp, direction).astype(np.complex128)
        ref = np.exp(direction * 2j * np.pi * ((j0 * k) % n) / n)
        assert fft_rel_err(X, np.broadcast_to(ref, X.shape)).max() <= tol(n)
        tone = np.exp(-direction * 2j * np.pi * ((f * k) % n) / n).astype(np.complex64)[None, :]
        Y = run_fft(bp, tone, direction)[0].astype(np.complex128)
        spike = np.zeros(n, np.complex128)
        spike[f] = n
        assert np.linalg.norm(Y - spike) / np.linalg.norm(spike) <= tol(n)
    x = si.fft_c64(3, n, stream=2200 + n)
    y = run_fft(bp, run_fft(bp, x, -1), +1).astype(np.complex128) / n
    assert fft_rel_err(y, x.astype(np.complex128)).max() <= 2 * tol(n)


def test_fft_mixed_radix_large_batch_sampled(bp):
    """A full-size batch (2^24 elements of n = 1000) checked on sampled signals."""
    n = 1000
    batch = (1 << 24) // n
    x = si.fft_c64(batch, n, stream=1999)
    X = run_fft(bp, x, -1)
    rows = np.unique(np.random.default_rng(4).integers(0, batch, 24))
    assert fft_rel_err(X[rows], oracle.dft(x[rows], -1)).max() <= tol(n)


@pytest.mark.parametrize("n", [375, 3000])
def test_fft_mixed_radix_round_trip_in_place(bp, n):
    batch = 5
    x = si.fft_c64(batch, n, stream=2100 + n)
    t = c64_to_dev(x.reshape(-1))
    bp.fft_batched(t, t, n, batch, -1)
    bp.fft_batched(t, t, n, batch, +1)
    torch.cuda.synchronize()
    y = c64_from_dev(t).reshape(batch, n) / n
    assert fft_rel_err(y, x.astype(np.complex128)).max() <= 2 * tol(n)


def test_fft_bluestein_round_trip_and_in_place(bp):
    n, batch = 1000, 4
    x = si.fft_c64(batch, n, stream=901)
    t = c64_to_dev(x.reshape(-1))
    bp.fft_batched(t, t, n, batch, -1)
    bp.fft_batched(t, t, n, batch, +1)
    torch.cuda.synchronize()
    y = c64_from_dev(t).reshape(batch, n) / n
    assert fft_rel_err(y, x.astype(np.complex128)).max() <= 2 * tol(n)


@pytest.mark.parametrize("n", [100003, 1 << 20 | 1, (1 << 23) - 1])
def test_fft_bluestein_large_closed_forms(bp, n):
    # an impulse at j0 gives exp(-2 pi i j0 k / n); a tone at f gives n at f
    k = np.arange(n, dtype=np.float64)
    j0, f = 12345, 777
    imp = np.zeros((1, n), np.complex64)
    imp[0, j0] = 1
    X = run_fft(bp, imp, -1)[0].astype(np.complex128)
    ref = np.exp(-2j * np.pi * ((j0 * k) % n) / n)
    assert np.linalg.norm(X - ref) / np.linalg.norm(ref) <= tol(n)
    tone = np.exp(2j * np.pi * ((f * k) % n) / n).astype(np.complex64)[None, :]
    Y = run_fft(bp, tone, -1)[0].astype(np.complex128)
    spike = np.zeros(n, np.complex128)
    spike[f] = n
    assert np.linalg.norm(Y - spike) / np.linalg.norm(spike) <= tol(n)


def test_fft_bluestein_inner_plan(bp):
    n, batch = 300, 4
    M = next_pow2(2 * n - 1)
    x = si.fft_c64(batch, n, stream=902)
    ref = oracle.dft(x, -1)
    for p in bp.enumerate_plans(bp.OP_FFT, bp.F32, M)[::7]:
        assert fft_rel_err(run_fft(bp, x, -1, p), ref).max() <= tol(n), p
    with pytest.raises(bp.BplgError):
        run_fft(bp, x, -1, bp.enumerate_plans(bp.OP_FFT, bp.F32, 2 * M)[0])  # not made for M
