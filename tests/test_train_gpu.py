"""Training kernels at the edges of their tiles: loss and gradient of the tcgen05 engine against the
mma.sync engine, and a fit with and without its loss history."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim  # noqa: E402

pytestmark = pytest.mark.gpu

# the layers' ranges in the flat parameters: W, b of layers 1-4
_SIZES = [12 * 256, 256, 256 * 256, 256, 256 * 256, 256, 256 * 4, 4]


def _data(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.normal(size=(n, 12)).astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
            (rng.random((n, 4)) < 0.8).astype(np.float32))


@pytest.mark.parametrize("n", [1, 100, 128, 129, 257, 1000, 16_384, 16_421])
def test_gradient_matches_the_other_engine(n):
    """Both engines round the same BF16 operands and differ in the order of FP32 sums (2^-24 each, sums
    of up to 16 421 terms) and where that moves a hidden unit over a BF16 rounding boundary (2^-8 of one
    value, about one in 2^13): far below 2e-3 of a layer's gradient norm."""
    X, T, M = _data(n, n)
    M[0, 0] = 1.0
    m = casim.casim_mlp_create(seed=5)
    try:
        got = {}
        for engine in (1, 0):
            casim.casim_mlp_set_engine(m, engine)
            got[engine] = casim.casim_mlp_loss_grad_host(m, X, T, M)
    finally:
        casim.casim_mlp_free(m)
    assert abs(got[1][0] - got[0][0]) <= 2e-3 * got[0][0]
    at = 0
    for size in _SIZES:
        a, b = got[1][1][at:at + size], got[0][1][at:at + size]
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b), (n, at)
        at += size


@pytest.mark.parametrize("batch", [1, 129, 3000])
def test_fit_is_the_same_with_and_without_history(batch):
    n = 4000
    X, Y, M = (torch.from_numpy(a).cuda() for a in _data(n, 3))
    params = []
    for history in (True, False):
        m = casim.casim_mlp_create(seed=6)
        try:
            hist = casim.casim_mlp_fit(m, X, Y, M, n, 3, batch, 1e-3, 9, history=history)
            if history:
                assert hist.shape == (3,) and np.isfinite(hist).all()
            params.append(casim.casim_mlp_get_params(m))
        finally:
            casim.casim_mlp_free(m)
    assert np.array_equal(params[0], params[1])
