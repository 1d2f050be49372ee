"""The one-launch LSQR loop of small systems: the shared memory of its
instrumental x at the limits of its sizes."""
import numpy as np
import pytest

import oracle
from paper_2212_11675_gb300 import _lib, gen
from tests.test_gpu_forms import _random

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def _solver(sys, **kw):
    from paper_2212_11675_gb300.solver import Solver
    return Solver(sys, **kw)


# 16 bytes an instrument beside the kernel's static shared memory: 3,024 end
# within the 48 KB of a launch that asks for nothing, 3,072 are the split
# form's limit
@pytest.mark.parametrize("n_instr", [3024, 3025, 3072, 3073])
@pytest.mark.parametrize("precision", [_lib.GSR_PREC_FP64, _lib.GSR_PREC_MIXED])
def test_instruments_at_the_shared_memory_limit(n_instr, precision):
    sys = _random(300, 12, 50, n_instr, seed=3)
    b = oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4)
    ref = oracle.pc_lsqr(sys, b, 12, 0.0, 0.0)
    with _solver(sys, precision=precision) as s:
        x, _, res = s.lsqr_solve(torch.tensor(b, device=DEV), 12, 0.0, 0.0)
        assert res["itn"] == ref["itn"] == 12
        assert np.linalg.norm(x.cpu().numpy() - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])
        assert s.kernel_status() == _lib.GSR_OK
