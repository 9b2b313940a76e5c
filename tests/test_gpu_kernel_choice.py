"""Each rule that chooses a kernel, on both sides of its line, against the oracle."""

import numpy as np
import pytest

from oracle import oracle as O
from synth import Workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_16892_gb300 import kvdro  # noqa: E402
from paper_2607_16892_gb300.runner import run  # noqa: E402
from tests.parity import compare_full  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def make(classes, L, r, lam, eps, cp, cw):
    classes = [np.asarray(c, np.int32) for c in classes]
    off = np.zeros(len(classes) + 1, np.int64)
    off[1:] = np.cumsum([len(c) for c in classes])
    K = len(classes)
    arr = lambda v: np.atleast_1d(np.asarray(v, np.float64))  # noqa: E731
    return Workload(name="choice", samples=np.concatenate(classes), offsets=off, L=np.full(K, L, np.int32),
                    L_in=np.zeros(K, np.int32), r=np.asarray(r, np.int32), lam=arr(lam), eps=arr(eps), cp=arr(cp),
                    cw=arr(cw), fractiles=arr([0.5]))


@pytest.mark.parametrize("L,cost", [(900, 3.0), (1 << 22, 3.0), ((1 << 22) + 1, 3.0), (900, 1e294), (900, 1e295),
                                    (900, 1e296)])
def test_fp64_requests(L, cost):
    """The exact kernel up to a support of 2^22 and a cost times L N of 1e300 (2.2e294 here), native
    FP64 above either.  Both hold the FP64 tolerance; where the exact kernel serves the request the
    results are its own, bit for bit."""
    rng = np.random.default_rng(5)
    w = make([rng.integers(0, L + 1, 500), rng.integers(0, 60, 33)], L, [0, 5, L // 2, L], cost * np.logspace(-3, 1, 21),
             [0.0, 3.0, 50.0], [cost, cost / 7], [cost / 3, cost])
    got = run(w, kvdro.KVDRO_FP64)
    compare_full(w, got, O.solve(w), "fp64")
    if L <= 1 << 22:
        same = all(np.array_equal(v, got[k]) for k, v in run(w, kvdro.KVDRO_EXACT).items())
        assert same or cost > 2e294


@pytest.mark.parametrize("nl", [1, 2, 3, 31, 32, 33, 64, 101, 256])
@pytest.mark.parametrize("order", ["ascending", "shuffled", "repeated"])
def test_envelope_lam_grids(nl, order):
    """Lanes along lam and rows of r per warp (widths 1 to 32), the saturated tail of an ascending grid that
    is not evaluated, and the FP32 look at the minimum over lam, against the exact kernel's results: the same
    integer sums and roundings, so every output is the same bit for bit, lowest-index ties included."""
    rng = np.random.default_rng(nl)
    lam = np.logspace(-3, 2, nl)
    if order == "shuffled":
        rng.shuffle(lam)
    elif order == "repeated":
        lam = np.repeat(lam, 2)[:nl]
    w = make([rng.integers(0, 4001, 700), rng.integers(0, 90, 41)], 4000, np.unique(rng.integers(0, 4001, 83)), lam,
             np.concatenate([[0.0], np.logspace(0, 3, 1 + nl % 17)]), [10.0, 0.5, 0.0], [1.0, 2.0, 1.0])
    exact, env = run(w, kvdro.KVDRO_EXACT), run(w, kvdro.KVDRO_ENVELOPE)
    for key, v in exact.items():
        assert np.array_equal(v, env[key]), key


@pytest.mark.parametrize("scale", [1e-150, 1e-32, 1e-25, 1e28, 1e33, 1e150])
def test_envelope_magnitudes(scale):
    """Costs and multipliers around the ends of what the FP32 look at a minimum takes (2^+-100, 2^-80)."""
    rng = np.random.default_rng(3)
    w = make([rng.integers(0, 901, 300)], 900, np.arange(0, 901, 25), scale * np.logspace(-3, 1, 40), [0.0, 1.0, 70.0],
             [10 * scale], [scale])
    exact, env = run(w, kvdro.KVDRO_EXACT), run(w, kvdro.KVDRO_ENVELOPE)
    for key, v in exact.items():
        assert np.array_equal(v, env[key]), key
    compare_full(w, env, O.solve(w), "fp64")


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 127, 128, 129, 4095, 4096, 4097, 8191, 8192, 8193, 24577])
@pytest.mark.parametrize("L,nl", [(1, 3), (300, 9), (1 << 19, 1), ((1 << 21) + 1, 9), (1 << 22, 1), (1 << 22, 9)])
def test_exact_quads(n, L, nl):
    """Quads of sorted samples (a class's last one starting with zeros, 8192 samples to a chunk) as integers
    up to 2^24 in float bit patterns: the sums of the exact and the envelope mode are the same integers,
    so every output is the same bit for bit.  Samples at 0 and at the top of the support, against
    reservations at both ends, make a lane's sums as large as they get between folds (6 loads at 2^22)."""
    rng = np.random.default_rng(n)
    x = rng.integers(0, L + 1, n)
    x[: n // 2] = L
    w = make([x], L, np.unique([0, 1, L // 3, L - 1, L]), np.logspace(-2, 2, nl), [0.0, 30.0], [10.0, 0.3], [1.0, 1.0])
    exact, env = run(w, kvdro.KVDRO_EXACT), run(w, kvdro.KVDRO_ENVELOPE)
    for key, v in exact.items():
        assert np.array_equal(v, env[key]), key


@pytest.mark.parametrize("L", [1, 2, 7, 400])
@pytest.mark.parametrize("cp,cw", [(10.0, 1.0), (1.0, 10.0), (3.0, 3.0), (5.0, 0.0), (0.0, 5.0), (0.0, 0.0), (1e6, 1.0),
                                   (1.0, 1e6)])
def test_dual_on_each_side_of_the_smaller_cost(L, cp, cw):
    """The search runs below min(c_p, c_w) or between the costs, over thresholds that rise or fall with gamma,
    with minima at 0, at the smaller cost, at the larger and between; every integer r, radii from 0 past L."""
    rng = np.random.default_rng(L)
    w = make([rng.integers(0, L + 1, 60), np.full(5, L), np.zeros(4)], L, np.arange(L + 1), [1.0],
             np.concatenate([[0.0], np.logspace(-3, np.log10(2.0 * L + 1.0), 37)]), cp, cw)
    ctx = kvdro.kvdro_create(0)
    try:
        kvdro.kvdro_load_samples(ctx, w.K, w.offsets, torch.from_numpy(w.samples).cuda(), w.L, w.L_in)
        shape = (1, len(w.eps), w.K, len(w.r))
        cost, gamma = np.empty(shape), np.empty(shape)
        kvdro.kvdro_eval_dual(ctx, len(w.r), w.r, len(w.eps), w.eps, 1, w.cp, w.cw, cost=cost, gamma=gamma)
    finally:
        kvdro.kvdro_destroy(ctx)
    ref = O.solve_dual(w)["cost"]
    size = cw * L + cp * L + max(cp, cw) * L  # the lines that cross at a minimiser are no larger
    assert np.all(np.abs(cost - ref) <= 1e-12 * np.abs(ref) + 16 * np.finfo(float).eps * size)
    assert np.all((gamma >= 0) & (gamma <= max(cp, cw)))


@pytest.mark.parametrize("nl", [9, 72, 100, 129, 200])
def test_exact_passes_over_the_samples(nl, monkeypatch):
    """CTAs whose rows take two to four passes (the chunk ring runs on across them, classes of one and of two
    chunks), against the envelope's same integers; and a bounded wait that runs out inside such a CTA."""
    rng = np.random.default_rng(nl)
    w = make([rng.integers(0, 3001, 9001), rng.integers(0, 400, 333)], 3000, np.arange(0, 3001, 3), np.logspace(-3, 2, nl),
             [0.0, 7.0, 90.0], [10.0, 4.0, 300.0], [1.0, 1.0, 1.0])
    outputs = ("cost", "lam_idx", "r_idx", "min_cost", "fhat")
    exact, env = run(w, kvdro.KVDRO_EXACT, outputs=outputs), run(w, kvdro.KVDRO_ENVELOPE, outputs=outputs)
    for key, v in exact.items():
        assert np.array_equal(v, env[key]), key
    monkeypatch.setenv("KVDRO_TEST_SKIP_CHUNK", "1")
    with pytest.raises(kvdro.KvdroError) as e:
        run(w, kvdro.KVDRO_EXACT, outputs=outputs, host_outputs=True)
    assert e.value.status == kvdro.KVDRO_ETIMEOUT


@pytest.mark.parametrize("L", [1, 31, 511, 513, 4095, 4096, 32766, 32895, 32896, 40961, 65534, 65535, 70000, 1 << 20])
@pytest.mark.parametrize("n", [1, 3, 127, 129, 4096, 4099, 70001])
def test_sort_supports_and_sizes(L, n):
    """Supports on and around the histogram's shared bins (2 x 16448), the scan's tiles (4096) and the tiles up
    to which it needs no pass of totals (16), class sizes around the expansion's steps and tiles, runs longer
    and shorter than a lane's four positions, a class whose offset is not a multiple of four, and one long run
    among single samples (tiles laid out in shared memory: 512 to 40960 bins)."""
    rng = np.random.default_rng(L + n)
    x = [rng.integers(0, L + 1, n), np.minimum(rng.geometric(0.3, n + 1), L), np.full(n, L),
         np.concatenate([np.full(n, L // 3), rng.integers(0, L + 1, n // 2 + 1)])]
    w = make(x, L, [0, L], [1.0], [0.0], 1.0, 1.0)
    got = run(w, kvdro.KVDRO_ENVELOPE, outputs=("sorted", "fhat", "S"))
    assert np.array_equal(got["sorted"], np.concatenate([np.sort(v) for v in x]))
    want = np.stack([[v.mean(), (L - v).mean()] for v in x])[None, :, :, None]  # at r = 0 and L, lam = 1 = c_p = c_w
    np.testing.assert_allclose(got["S"], want, rtol=1e-12)


MODES = {"fp32": kvdro.KVDRO_FP32, "fp64": kvdro.KVDRO_FP64, "exact": kvdro.KVDRO_EXACT, "envelope": kvdro.KVDRO_ENVELOPE}


def _tiny_factor_cases(L):
    """One factor of lam * eps below 2^-100, the other so large that the product decides the minimum."""
    rng = np.random.default_rng(8)
    at = np.full(40, 100)
    return [make([at], L, [L // 3, 2 * L // 3], [0.0, 7e-31], [1e3, 1e6], 1e-26, 1e-26),
            make([at], L, [L // 3, 2 * L // 3], [1e-32, 7e-31, 7.8e-31, 7.9e-31], [0.0, 1e2, 1e3, 1e6], [1e-26, 2e-26], [1e-26, 1e-26]),
            make([rng.integers(0, L + 1, 300)], L, [L // 2], [9.9995, 1e30], [7e-31], 10.0, 1.0),
            make([rng.integers(0, L + 1, 300)], L, [L // 4, L // 2], np.concatenate([np.linspace(9.99, 10.0, 30), [1e27, 1e30]]),
                 [0.0, 1e-300, 7e-31, 7.9e-31], 10.0, 1.0)]


@pytest.mark.parametrize("mode,L", [("fp32", 900), ("fp64", 900), ("exact", 900), ("envelope", 900),
                                    ("fp32", (1 << 22) + 3), ("fp64", (1 << 22) + 3), ("noalloc", 900)])
def test_products_of_a_tiny_and_a_large_factor(mode, L):
    """A lam or a radius that a float look at the minimum takes for zero still counts through its product
    with the other, in every kernel: exact, FP32 and FP64 arithmetic, envelope, and the allocation-free call."""
    from tests.test_zz_no_alloc import _noalloc
    for w in _tiny_factor_cases(L):
        got = _noalloc(w) if mode == "noalloc" else run(w, MODES[mode])
        compare_full(w, got, O.solve(w), "fp32" if mode in ("fp32", "noalloc") else "fp64")


@pytest.mark.parametrize("mode", ["fp32", "fp64", "exact", "envelope"])
def test_sums_past_the_double_range_leave_the_finite_ones(mode):
    """c_p so large that the class sums of small multipliers pass the double range: their S is infinite or not
    a number, and the minimum over lam is taken over the others, here from lam = c_p on, where 15 of the 500
    samples lie 1 to 5 above r."""
    x = np.concatenate([np.full(485, 10), np.repeat(np.arange(891, 896), 3)])
    w = make([x], 900, [890], [0.0, 1e290, 1e305, 2e305], [0.0], 1e305, 0.0)
    got = run(w, MODES[mode], outputs=("cost", "lam_idx", "r_idx", "min_cost"))
    assert got["lam_idx"].tolist() == [[[[2]]]] and got["r_idx"].tolist() == [[[0]]]
    if mode != "fp32":  # beyond FP32
        np.testing.assert_allclose([got["cost"].item(), got["min_cost"].item()], 1e305 / 500 * 45, rtol=1e-12)


def test_dual_values_past_the_double_range_are_not_the_empirical_cost():
    """The same samples at a radius that puts the minimiser at gamma = 0, where g = 1e306 and its class sum is past
    the double range: the result is no number, or the value, but not the empirical cost of 9e303 below it."""
    x = np.concatenate([np.full(485, 10), np.repeat(np.arange(891, 896), 3)])
    ctx = kvdro.kvdro_create(0)
    try:
        kvdro.kvdro_load_samples(ctx, 1, np.array([0, 500]), torch.from_numpy(x.astype(np.int32)).cuda(), [900])
        cost = np.empty((1, 1, 1, 1))
        kvdro.kvdro_eval_dual(ctx, 1, [890], 1, [1e6], 1, [1e305], [0.0], cost=cost)
    finally:
        kvdro.kvdro_destroy(ctx)
    assert np.isnan(cost.item()) or abs(cost.item() - 1e306) <= 1e-12 * 1e306


@pytest.mark.parametrize("mode,L", [("fp32", 1000), ("exact", 1000), ("fp32", (1 << 22) + 1), ("fp64", (1 << 22) + 1)])
def test_rows_after_a_wait_that_runs_out(mode, L, monkeypatch):
    """With the first chunk's copy left out every CTA of the exact kernel, and above 2^22 of the FP32- and
    FP64-arithmetic kernels, gives up: no r was evaluated, and r_idx says so (-1) whether the rows are
    finalised by the last CTA or by a launch.  With the second, the classes of one chunk have their results."""
    rng = np.random.default_rng(3)
    w = make([rng.integers(0, 900, 20000), rng.integers(0, 900, 77)], L, [10, 200, 600], [0.5, 5.0], [0.0, 10.0], 10.0, 1.0)
    ref = O.solve(w)
    for skip in (0, 1):
        monkeypatch.setenv("KVDRO_TEST_SKIP_CHUNK", str(skip))
        ctx = kvdro.kvdro_create(0)
        monkeypatch.delenv("KVDRO_TEST_SKIP_CHUNK")
        try:
            kvdro.kvdro_load_samples(ctx, w.K, w.offsets, torch.from_numpy(w.samples).cuda(), w.L, w.L_in)
            r_idx = torch.full((1, 2, 2), 7, dtype=torch.int32, device="cuda")
            kvdro.kvdro_eval_grid(ctx, MODES[mode], 3, w.r, 2, w.lam, 2, w.eps, 1, w.cp, w.cw, r_idx=r_idx)
            with pytest.raises(kvdro.KvdroError) as e:
                kvdro.kvdro_sync(ctx)
            assert e.value.status == kvdro.KVDRO_ETIMEOUT
        finally:
            kvdro.kvdro_destroy(ctx)
        got = r_idx.cpu().numpy()[0]
        assert np.all(got[:, 0] == -1)
        assert np.array_equal(got[:, 1], ref["r_idx"][0, :, 1] if skip else [-1, -1])


@pytest.mark.parametrize("sizes", [(4095, 4097), (8193,), (8191, 12289), (3, 3 * 4096 + 4093, 5 * 4096 + 2)])
def test_native_fp64_on_quads_over_several_chunks(sizes):
    """Costs past the exact kernel's bound run native FP64 on staged quads: samples taken back from them in
    every chunk of a ring of two, class sizes on either side of a chunk and of a quad."""
    rng = np.random.default_rng(sum(sizes))
    w = make([rng.integers(0, 901, n) for n in sizes], 900, [0, 5, 450, 899, 900], 1e296 * np.logspace(-3, 1, 21), [0.0, 3.0, 50.0],
             [1e296, 1e295], [3e295, 1e296])
    compare_full(w, run(w, kvdro.KVDRO_FP64), O.solve(w), "fp64")


@pytest.mark.parametrize("blocks", [255, 256, 257, 514])
def test_rows_finalised_by_the_last_cta_and_by_a_launch(blocks):
    """4 classes x 2 regimes x `blocks` CTAs of the exact kernel, up to 2048 of them finalised by the last CTA of
    each (regime, class), above by a launch, against the envelope, half as many CTAs."""
    rng = np.random.default_rng(blocks)
    w = make([rng.integers(0, 3001, n) for n in (300, 77, 4, 1)], 3000, np.arange(4 * blocks), np.logspace(-3, 2, 64),
             [0.0, 7.0, 90.0], [10.0, 4.0], [1.0, 1.0])
    outputs = ("cost", "lam_idx", "r_idx", "min_cost", "fhat")
    exact, env = run(w, kvdro.KVDRO_EXACT, outputs=outputs), run(w, kvdro.KVDRO_ENVELOPE, outputs=outputs)
    for key, v in exact.items():
        assert np.array_equal(v, env[key]), key
