"""A fit on a stream of its own while another thread keeps the default stream busy: the parameters of a
fit on the default stream, bit for bit.  (The first fit of a network makes its workspace: nothing in it
may be prepared on another stream than the one that trains.)"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [1, 0])
def test_fit_on_a_side_stream(engine):
    n, batch, steps = 20_000, 4096, 200
    rng = np.random.default_rng(4)
    X, Y, M = (torch.from_numpy(a.astype(np.float32)).cuda()
               for a in (rng.normal(size=(n, 12)), rng.normal(size=(n, 4)), rng.random((n, 4)) < 0.8))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    params = []
    for stream in (None, side):
        m = casim.casim_mlp_create(seed=8)
        done = threading.Event()

        def busy():
            while not done.is_set():
                # some 1.5 ms each: what is queued behind them would run in the middle of the fit
                torch.cuda._sleep(3_000_000)
                torch.cuda._sleep(3_000_000)
                torch.cuda.default_stream().synchronize()

        thread = threading.Thread(target=busy)
        try:
            casim.casim_mlp_set_engine(m, engine)
            torch.cuda.synchronize()
            if stream is not None:
                thread.start()
            casim.casim_mlp_fit(m, X, Y, M, n, steps, batch, 1e-3, 9, stream=stream, history=False)
        finally:
            done.set()
            if stream is not None:
                thread.join()
            params.append(casim.casim_mlp_get_params(m))
            casim.casim_mlp_free(m)
    assert np.isfinite(params[0]).all()
    assert np.array_equal(params[0], params[1])
