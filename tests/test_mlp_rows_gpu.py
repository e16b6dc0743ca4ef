"""The tensor-core network over row counts at the edges of its tiles and of its two tiles in flight.

A row's result does not depend on the rows beside it: every count, and every offset of the rows in
the tiles, gives the same bits as the widest call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim  # noqa: E402

pytestmark = pytest.mark.gpu


def test_rows_do_not_depend_on_the_tiling():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wave = 128 * sms                       # one tile per CTA
    total = 4 * wave + 77
    m = casim.casim_mlp_create(seed=7)
    try:
        X = torch.randn((total, 12), generator=torch.Generator().manual_seed(3), dtype=torch.float32).cuda()

        def run(x):
            y = torch.full((x.shape[0], 4), float("nan"), dtype=torch.float32, device="cuda")
            casim.casim_mlp_forward(m, x, y)
            return y.cpu().numpy()

        want = run(X)
        assert np.isfinite(want).all()
        for n in (1, 127, 128, 129, wave - 1, wave, wave + 1, 2 * wave, 2 * wave + 1, 3 * wave - 5, 3 * wave + 129):
            for off in (0, 5):
                assert np.array_equal(run(X[off:off + n].contiguous()), want[off:off + n]), (n, off)
    finally:
        casim.casim_mlp_free(m)
