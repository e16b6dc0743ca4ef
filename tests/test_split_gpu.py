"""The split step (several threads per column, few columns) against the one-thread-per-column step.

The same columns give the same bits whether they are a domain of their own, whose levels are shared
by up to 32 threads, or the first columns of a domain wide enough for one thread per column."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import casim, synth  # noqa: E402

pytestmark = pytest.mark.gpu

W, A, Z = casim.CASIM_WARM, casim.CASIM_AEROSOL, casim.CASIM_THREE_MOMENT
FLAGS = {0: 16, W: 16, A: 22, W | A: 19, Z: 20, W | Z: 17}
WIDE = 80_000     # above one resident wave of warps for every configuration


def _fields(nf, ncols, nlev, dz, seed):
    base = synth.make_state("deep_convective", ncols, nlev, dz, seed=seed)
    fld = np.zeros((nf,) + base.shape[1:])
    fld[:16] = base
    rng = np.random.default_rng(seed)
    if nf in (19, 22):
        fld[16] = rng.uniform(1e-9, 5e-9, base.shape[1:])
        for f, q in zip(range(17, nf), (2, 3, 4, 5, 6)):
            fld[f] = base[q] * 1e-5
    elif nf > 16:     # shape 2: G = 6 7 8 / (3 4 5)
        for f, q, n, dens in zip(range(16, nf), (3, 4, 5, 6), (8, 9, 10, 11), (1000.0, 500.0, 100.0, 400.0)):
            ok = base[n] > 0
            fld[f][ok] = 5.6 * (base[q][ok] / (np.pi / 6 * dens)) ** 2 / base[n][ok]
    return fld


def _step(fld, dz, ncols, flags, precision, dt, tend):
    ctx = casim.casim_init(precision=precision, flags=flags)
    try:
        d = casim.Domain(fld, dz, ncols)
        out = d.fld
        if tend:
            out = torch.zeros((fld.shape[0] - 3,) + fld.shape[1:], dtype=torch.float64, device="cuda")
            casim.casim_step_tendency(ctx, d.state, ncols, d.nlev, dt, out)
        else:
            casim.casim_step(ctx, d.state, ncols, d.nlev, dt)
        rc, bits = casim.casim_get_error(ctx)
        assert (rc, bits) == (0, 0)
        return out[:, :, :ncols].cpu().numpy(), d.precip[:, :ncols].cpu().numpy()
    finally:
        casim.casim_free(ctx)


@pytest.mark.parametrize("precision", [casim.CASIM_MIXED, casim.CASIM_FP64])
@pytest.mark.parametrize("flags", list(FLAGS))
def test_split_step_equals_one_thread_per_column(flags, precision):
    for ncols, nlev in ((1, 1), (33, 2), (200, 7), (700, 70), (5000, 33)):
        dz = synth.dz_stretched(nlev)
        fld = _fields(FLAGS[flags], ncols, nlev, dz, seed=100 + nlev)
        wide = np.ascontiguousarray(np.tile(fld[:, :, :ncols], (1, 1, -(-WIDE // ncols)))[:, :, :WIDE])
        for dt, tend in ((1.0, False), (30.0, False), (2.0, True), (30.0, True)):
            a = _step(fld, dz, ncols, flags, precision, dt, tend)
            b = _step(wide, dz, WIDE, flags, precision, dt, tend)
            for x, y in zip(a, b):
                assert np.array_equal(x, y[..., :ncols]), (ncols, nlev, dt, tend)


@pytest.mark.parametrize("flags", list(FLAGS))
def test_blocks_of_64_threads_equal_blocks_of_128(flags):
    """One thread per column in at most one resident wave: blocks of half the size, same bits."""
    nlev = 13
    dz = synth.dz_stretched(nlev)
    base = _fields(FLAGS[flags], 700, nlev, dz, seed=31)
    wide = np.ascontiguousarray(np.tile(base, (1, 1, -(-WIDE // 700)))[:, :, :WIDE])
    for dt, tend in ((1.0, False), (30.0, False), (1.0, True), (30.0, True)):
        b = _step(wide, dz, WIDE, flags, casim.CASIM_MIXED, dt, tend)
        for ncols in (50_001, 65_536):
            fld = np.ascontiguousarray(wide[:, :, :-(-ncols // 32) * 32])
            a = _step(fld, dz, ncols, flags, casim.CASIM_MIXED, dt, tend)
            for x, y in zip(a, b):
                assert np.array_equal(x, y[..., :ncols]), (ncols, dt, tend)
