"""Bounded device waits that run out: the call says GSR_ERR_TIMEOUT soon (not
after a wait per iteration), and the handle works again.  Nothing faults and
nothing is left waiting: a copy is announced and never issued, a barrier waits
for an arrival or a block that does not come."""
import time

import numpy as np
import pytest

import oracle
from paper_2212_11675_gb300 import _lib, gen
from tests._dense import small

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def _system():
    sys = small(257, 37, 11, seed=31)
    return sys, torch.tensor(oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4), device=DEV)


def _solver(sys, **kw):
    from paper_2212_11675_gb300.solver import Solver
    return Solver(sys, **kw)


def _timeout(call):
    t0 = time.time()
    with pytest.raises(_lib.GsrError) as e:
        call()
    assert e.value.code == _lib.GSR_ERR_TIMEOUT
    return time.time() - t0


@pytest.mark.parametrize("kind", ["mixed", "batched", "batched two runs"])
def test_missing_copy_in_the_inner_loops(kind):
    sys, b = _system()
    k = {"mixed": 0, "batched": 8, "batched two runs": 9}[kind]
    B = b.repeat(k, 1) if k else b
    with _solver(sys, precision=_lib.GSR_PREC_MIXED, conlim=0.0) as s:
        def solve():
            return (s.batched_solve(B, 10, 100) if k else s.mixed_solve(B, 10, 100))[0].cpu().numpy()
        ref = solve()
        s.inject_missing_copy(1)
        # the waits of one iteration's passes and of the FP64 products around it
        assert _timeout(solve) < 10.0
        s.inject_missing_copy(-1)
        assert s.kernel_status() == _lib.GSR_OK
        x = solve()
        assert s.kernel_status() == _lib.GSR_OK
    assert np.linalg.norm(x - ref) <= 1e-12 * np.linalg.norm(ref)


def test_missing_copy_of_a_window():
    # 40,000 rows: window 0 is copied by the row-window pass, tile 0 by others
    sys = small(2000, 400, 60, seed=5)
    rng = np.random.default_rng(6)
    y = torch.tensor(rng.standard_normal(sys.m), device=DEV)
    with _solver(sys, precision=_lib.GSR_PREC_MIXED) as s:
        ref = s.aprod2_f32(y, torch.zeros(s.n, dtype=torch.float64, device=DEV)).cpu().numpy()
        s.inject_missing_copy(0)
        s.aprod2_f32(y, torch.zeros(s.n, dtype=torch.float64, device=DEV))
        assert s.kernel_status() == _lib.GSR_ERR_TIMEOUT
        s.inject_missing_copy(-1)
        x = s.aprod2_f32(y, torch.zeros(s.n, dtype=torch.float64, device=DEV)).cpu().numpy()
        assert s.kernel_status() == _lib.GSR_OK
    assert np.array_equal(x, ref)


def test_missing_copy_ends_the_lsqr_and_cg_iterations():
    sys, b = _system()
    g = torch.tensor(np.random.default_rng(7).standard_normal(sys.n), device=DEV)
    with _solver(sys, conlim=0.0) as s:
        s.inject_missing_copy(1)
        assert _timeout(lambda: s.lsqr_solve(b, 200, 0.0, 0.0)) < 10.0
        assert _timeout(lambda: s.normal_solve(g, 200, 0.0)) < 10.0
        s.inject_missing_copy(-1)
        q, info = s.normal_solve(g)
        assert info["converged"] == 1 and s.kernel_status() == _lib.GSR_OK


def test_missing_block_in_the_one_launch_loop():
    sys, b = _system()
    ref = oracle.pc_lsqr(sys, b.cpu().numpy(), 12, 0.0, 0.0)["x"]
    with _solver(sys) as s:
        assert s.lsqr_one_launch()
        s.inject_missing_block(1)
        assert _timeout(lambda: s.lsqr_solve(b, 12, 0.0, 0.0)) < 10.0
        s.inject_missing_block(0)
        x, _, res = s.lsqr_solve(b, 12, 0.0, 0.0)
        assert res["itn"] == 12 and s.kernel_status() == _lib.GSR_OK
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
