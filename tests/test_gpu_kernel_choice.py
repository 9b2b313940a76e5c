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
