"""Mixed warm configurations with a third field: substeps beyond a pass of 16 (one thread per column)
give the bits of one pass of all (the split step)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim, synth  # noqa: E402

pytestmark = pytest.mark.gpu

WIDE = 160_000     # one thread per column in every warm configuration


@pytest.mark.parametrize("dt", [10.0, 50.0, 90.0, 200.0])
@pytest.mark.parametrize("names,nf", [(("CASIM_WARM", "CASIM_AEROSOL"), 19), (("CASIM_WARM", "CASIM_THREE_MOMENT"), 17)])
def test_passes(names, nf, dt):
    """Layers of 40 m and a capped speed of 10 m/s or so: from 3 substeps to the cap of 64."""
    flags = sum(getattr(casim, n) for n in names)
    nlev, ncols = 24, 640
    dz = np.full(nlev, 40.0)
    base = synth.make_state("deep_convective", ncols, nlev, dz, seed=23)
    fld = np.zeros((nf,) + base.shape[1:])
    fld[:16] = base
    if nf == 19:
        fld[16], fld[17], fld[18] = 2e-9, base[2] * 1e-5, base[3] * 1e-5
    else:
        ok = base[8] > 0
        fld[16][ok] = 9.0 * (base[3][ok] / (np.pi / 6 * 1000.0)) ** 2 / base[8][ok]
    wide = np.ascontiguousarray(np.tile(fld[:, :, :ncols], (1, 1, WIDE // ncols)))
    outs = []
    for f, n in ((fld, ncols), (wide, WIDE)):
        ctx = casim.casim_init(precision=casim.CASIM_MIXED, flags=flags)
        try:
            d = casim.Domain(f, dz, n)
            casim.casim_step(ctx, d.state, n, nlev, dt)
            assert casim.casim_get_error(ctx)[1] & ~2 == 0      # bit 1: more substeps wanted than the cap
            outs.append((d.fld[:, :, :ncols].cpu().numpy(), d.precip[:, :ncols].cpu().numpy()))
        finally:
            casim.casim_free(ctx)
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
