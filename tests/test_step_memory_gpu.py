"""A step takes no device memory of its own: the kernels' local memory fits what the context has set
aside for every thread (a larger stack makes the device reserve more at the first launch, and keep it)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_CODE = """
import sys
import numpy as np, torch
from paper_2010_14823_gb300 import casim, synth
precision, flags, nf = (int(x) for x in sys.argv[1:])
nlev = 20
dz = synth.dz_stretched(nlev)
base = synth.make_state("deep_convective", 256, nlev, dz, seed=1)
fld = np.zeros((nf,) + base.shape[1:])
fld[:16] = base
ctx = casim.casim_init(precision=precision, flags=flags)
d = casim.Domain(fld, dz, 256)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
casim.casim_step(ctx, d.state, 256, nlev, 1.0)
torch.cuda.synchronize()
print(free - torch.cuda.mem_get_info()[0])
casim.casim_free(ctx)
"""


@pytest.mark.parametrize("precision", ["CASIM_FP64", "CASIM_MIXED"])
@pytest.mark.parametrize("names,nf", [((), 16), (("CASIM_STATS",), 16), (("CASIM_AEROSOL",), 22), (("CASIM_THREE_MOMENT",), 20)])
def test_first_step_takes_no_memory(precision, names, nf):
    from paper_2010_14823_gb300 import casim
    flags = sum(getattr(casim, n) for n in names)
    out = subprocess.run([sys.executable, "-c", _CODE, str(getattr(casim, precision)), str(flags), str(nf)],
                         cwd=ROOT, check=True, capture_output=True, text=True).stdout
    assert int(out.split()[-1]) == 0
