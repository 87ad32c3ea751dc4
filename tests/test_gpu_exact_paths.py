"""Exact-arithmetic paths of mixed plans at the edges of their tiles, against the FP64 oracle.

Tolerances come from the arithmetic, stated at each test.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.pinv_oracle as O  # noqa: E402
from paper_2410_06129_gb300 import _lib as L  # noqa: E402
from paper_2410_06129_gb300 import synth  # noqa: E402
from tests._ref import rel  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_tc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not L.load().pinv_tc_available():
        pytest.skip("tcgen05 kernels need sm_103a")


def _plan(*a, **kw):
    from paper_2410_06129_gb300.plan import Plan
    kw.setdefault("precision", L.MIXED_BF16X6)
    return Plan(*a, **kw)


@pytest.mark.parametrize("dims,coils", [((1,), 1), ((31,), 9), ((4, 8), 3), ((11, 3), 8), ((5, 4, 5), 17)])
def test_factored_gram_is_the_exact_gram(dims, coils):
    """Plans that keep the exact Gram factor it: N = 1, 31, 32, 33 and 100 (below, at and past a
    32-wide tile), coil counts below, at and past the 8 staged at a time. The kept Gram's lower
    triangle is the exported exact Gram's to an ulp, and both equal E^H E + lambda I to 1e-13
    (the exact Gram's own bar: double-float sums, 2^-45)."""
    rng = np.random.default_rng(31)
    N, D = int(np.prod(dims)), len(dims)
    k = rng.uniform(-0.5 * max(dims), 0.5 * max(dims), size=(3 * N + 1, D))
    maps = None
    if coils > 1:
        maps = rng.standard_normal((coils, N)) + 1j * rng.standard_normal((coils, N))
    E = O.encode(k, O.voxel_positions(dims), maps, None, None) if coils > 1 else O.encode(k, O.voxel_positions(dims))
    lam = O.lambda_abs(E, 1e-3)
    pl = _plan(dims, k, maps, lam=1e-3, keep_gram=True).build()
    G = np.tril(pl.export(L.EXPORT_GRAM).cpu().numpy())
    X = pl.export(L.EXPORT_GRAM_EXACT).cpu().numpy()
    want = E.conj().T @ E + lam * np.eye(N)
    assert rel(X, want) < 1e-13
    # the kept Gram joins the pairs on the integer pipe, the export on the FP64 pipe: one ulp
    assert rel(G, np.tril(X)) < 4e-16
    assert np.array_equal(X, X.conj().T)
