"""FP64 form: a condensate or number that is not a number counts as absent, whatever the NaN's sign."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2010_14823_gb300 import casim, synth  # noqa: E402

pytestmark = pytest.mark.gpu

F = {n: i for i, n in enumerate(synth.FIELDS)}
NAN = np.array([0x7FF8000000000000, 0xFFF8000000000000, 0x7FF0000000000001], dtype=np.uint64).view(np.float64)


@pytest.mark.parametrize("field", ["qc", "qr", "qi", "qs", "qg", "nc", "nr", "ni", "ns", "ng"])
def test_nan_stays_where_the_oracle_leaves_it(field):
    """One NaN in every fourth column, in clear air and in cloud: NaN afterwards where the oracle, whose
    comparisons are the language's, has NaN, and nowhere else; the step reports it."""
    ncols, nlev = 384, 60
    dz = synth.dz_stretched(nlev)
    fld = synth.make_state("deep_convective", ncols, nlev, dz, seed=12)
    rng = np.random.default_rng(5)
    for i, c in enumerate(range(0, ncols, 4)):
        fld[F[field], rng.integers(nlev), c] = NAN[i % 3]
    ref = fld.copy()
    oracle.step(ref, ncols, dz, 1.0)
    ctx = casim.casim_init(precision=casim.CASIM_FP64)
    try:
        d = casim.Domain(fld, dz, ncols)
        casim.casim_step(ctx, d.state, ncols, nlev, 1.0)
        rc, flags = casim.casim_get_error(ctx)
        out, _ = d.numpy()
    finally:
        casim.casim_free(ctx)
    assert (rc, flags) == (-4, 1)   # CASIM_ERR_NONFINITE
    for f in range(casim.NPROG):
        if field == "nc" and f == F["na"]:
            # activation leaves a point whose particle number is not a number alone; the oracle's goes on
            assert np.isfinite(out[f, :, :ncols]).all()
            continue
        a, b = np.isnan(out[f, :, :ncols]), np.isnan(ref[f, :, :ncols])
        assert np.array_equal(a, b), (synth.FIELDS[f], int(a.sum()), int(b.sum()))
