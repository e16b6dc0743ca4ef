"""FP64 form: points at and around saturation are taken up exactly where the oracle takes them up."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2010_14823_gb300 import casim, synth  # noqa: E402

pytestmark = pytest.mark.gpu

F = {n: i for i, n in enumerate(synth.FIELDS)}
# relative distances from saturation: outside, at and inside the FP32 decision's margin of 1e-4, and 1e-12
# (the two FP64 evaluations of q_s agree to 1e-14)
DIST = [s * d for d in (0.3, 1e-3, 1.1e-4, 1.01e-4, 1e-4, 0.99e-4, 9e-5, 1e-5, 1e-8, 1e-12) for s in (1, -1)]


def _qs(P, T, p, ice):
    if ice:
        es = P.es_i0 * np.exp(P.es_ia * (T - P.es_it) / (T - P.es_ib))
    else:
        es = P.es_l0 * np.exp(P.es_la * (T - P.T0) / (T - P.T0 + P.es_lb))
    eps = P.Rd / P.Rv
    return eps * es / (p - (1 - eps) * es), es


@pytest.mark.parametrize("ice", [False, True])
def test_points_around_saturation(ice):
    """Clear points from 70 K to above the boiling point, 1 hPa to 1100 hPa, and points whose pressure is
    within 1e-6 of (1 - eps) es, where q_s changes sign: a point is changed (condensation or nucleation)
    exactly where the oracle changes it."""
    P = casim.casim_default_params()
    rng = np.random.default_rng(9)
    nlev, ncols = len(DIST), 4096
    T = rng.uniform(70.0, 260.0 if ice else 360.0, (nlev, ncols))
    T[:, :64] = np.linspace(126.0, 130.0, 64)          # the FP32 decision's lower bound
    p = np.exp(rng.uniform(np.log(1e2), np.log(1.1e5), (nlev, ncols)))
    qs, es = _qs(P, T, p, ice)
    if not ice:
        c = slice(ncols - 256, ncols)
        T[:, c] = rng.uniform(340.0, 360.0, (nlev, 256))
        es = _qs(P, T, p, False)[1]
        p[:, c] = ((1 - P.Rd / P.Rv) * es * (1 + rng.choice([-1e-6, 1e-6, 1e-3, 1.0], (nlev, ncols))))[:, c]
        qs, es = _qs(P, T, p, False)
    dz = np.full(nlev, 100.0)
    fld = np.zeros((16, nlev, synth.pad_columns(ncols)))
    fld[F["T"], :, :ncols], fld[F["p"], :, :ncols] = T, p
    fld[F["rho"], :, :ncols] = p / (287.04 * T)
    qv = qs * (1 + np.array(DIST)[:, None])
    fld[F["qv"], :, :ncols] = np.where((qv > 0) & (qv < 0.05), qv, 0.02)
    ref = fld.copy()
    oracle.step(ref, ncols, dz, 1.0)
    ctx = casim.casim_init(precision=casim.CASIM_FP64)
    try:
        d = casim.Domain(fld, dz, ncols)
        casim.casim_step(ctx, d.state, ncols, nlev, 1.0)
        out, _ = d.numpy()
    finally:
        casim.casim_free(ctx)
    f = [F[n] for n in ("T", "qv", "qc", "qi", "ni")]
    got, want = ((x[f] != fld[f]).any(axis=0)[:, :ncols] for x in (out, ref))
    assert want.any() and not want.all()
    assert np.array_equal(got, want), (int((got != want).sum()), T[got != want][:5], p[got != want][:5])
