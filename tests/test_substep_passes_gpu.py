"""FP64 form with a third field per species: substeps beyond one pass of 32 against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim, synth  # noqa: E402

pytestmark = pytest.mark.gpu

F = {n: i for i, n in enumerate(synth.FIELDS)}


@pytest.mark.parametrize("dt", [30.0, 60.0, 120.0, 200.0])
def test_aerosol_standard_fields_are_the_cold_steps(dt):
    """Layers of 50 m and capped speeds of up to 20 m/s: some 12, 24, 48 and 64 (the cap) substeps.  The
    aerosol configuration takes 32 a pass, the standard one all: the fields they share are the same bits,
    and its aerosol is the column's but for what the surface row says (64 substeps of sums of 1e-16)."""
    ncols, nlev = 160, 40
    dz = np.full(nlev, 50.0)
    base = synth.make_state("deep_convective", ncols, nlev, dz, seed=17)
    fld = np.zeros((22,) + base.shape[1:])
    fld[:16] = base
    fld[16, :, :ncols] = 2e-9
    for f, q in zip(range(17, 22), (2, 3, 4, 5, 6)):
        fld[f] = base[q] * 1e-5
    outs = {}
    for flags, nf in ((0, 16), (casim.CASIM_AEROSOL, 22)):
        ctx = casim.casim_init(precision=casim.CASIM_FP64, flags=flags)
        try:
            d = casim.Domain(np.ascontiguousarray(fld[:nf]), dz, ncols)
            casim.casim_step(ctx, d.state, ncols, nlev, dt)
            rc, bits = casim.casim_get_error(ctx)
            assert bits & ~2 == 0      # bit 1: more substeps wanted than the cap
            outs[nf] = d.numpy()
        finally:
            casim.casim_free(ctx)
    assert np.array_equal(outs[22][0][:16], outs[16][0]) and np.array_equal(outs[22][1][:4], outs[16][1])
    w = fld[F["rho"], :, :ncols] * dz[:, None]
    before, after = ((x[16:22, :, :ncols] * w).sum(axis=(0, 1)) for x in (fld, outs[22][0]))
    lost = outs[22][1][4, :ncols]
    assert np.abs(before - after - lost).max() <= 64 * nlev * 2.0**-52 * before.max()
