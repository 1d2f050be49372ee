"""The one-launch LSQR loop of small systems: the shared memory of its
instrumental x at the limits of its sizes, and the systems it is taken for."""
import numpy as np
import pytest

import oracle
from paper_2212_11675_gb300 import _lib, gen
from tests._systems import drop_stars
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


# (stars, rows a star, knots, instruments), empty stars, one launch?  The lines
# lie at 75,000 rows, 60,000 columns and offsets of 16 pieces of 512 rows
@pytest.mark.parametrize("shape,empty,one", [
    ((2500, 30, 60, 30), 0, True), ((2500, 30, 60, 30), 1, True), ((2501, 30, 60, 30), 0, False),
    ((11951, 3, 61, 61), 0, True), ((11952, 3, 61, 61), 0, False),   # 60,000 and 60,005 columns
    ((12000, 5, 60, 30), 11000, False),                              # mostly empty stars
    ((512, 16, 4, 30), 0, True), ((513, 16, 4, 30), 0, False)])      # one offset: 16 and 17 pieces
def test_where_the_loop_is_taken(shape, empty, one):
    sys = _random(*shape, seed=9)
    if empty:
        sys = drop_stars(sys, range(1, 1 + empty))
    b = oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4)
    ref = oracle.pc_lsqr(sys, b, 5, 0.0, 0.0)
    with _solver(sys) as s, _solver(sys, eager=True) as e:
        assert s.lsqr_one_launch() is one and not e.lsqr_one_launch()
        x, se, res = s.lsqr_solve(torch.tensor(b, device=DEV), 5, 0.0, 0.0)
        assert res["itn"] == ref["itn"] == 5
        assert np.linalg.norm(x.cpu().numpy() - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])
        np.testing.assert_allclose(se.cpu().numpy(), ref["se"], rtol=1e-9)
        assert s.kernel_status() == _lib.GSR_OK
