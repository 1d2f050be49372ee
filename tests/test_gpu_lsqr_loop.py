"""The one-launch LSQR loop of small systems: the shared memory of its
instrumental x at the limits of its sizes, the systems it is taken for, and
solves beside other work on the GPU."""
import threading
import time

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
# lie at rows + 6 columns = 460,000 and offsets of 16 pieces of 512 rows
@pytest.mark.parametrize("shape,empty,one", [
    ((2000, 199, 100, 30), 0, True), ((2000, 199, 100, 30), 1, True),  # 459,986 without empty stars
    ((2000, 199, 100, 33), 0, False),                                  # 460,004
    ((13900, 3, 30, 30), 0, True), ((13920, 3, 30, 30), 0, False),     # 459,426 and 460,086
    ((16000, 5, 60, 30), 15000, False),                                # mostly empty stars
    ((512, 16, 4, 30), 0, True), ((513, 16, 4, 30), 0, False)])        # one offset: 16 and 17 pieces
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


def test_solve_beside_a_kernel_that_holds_an_sm():
    # one block of another stream for about 1.2 s on an SM that the loop needs too
    sys = _random(257, 20, 37, 11, seed=9)
    b = oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4)
    ref = oracle.pc_lsqr(sys, b, 12, 0.0, 0.0)
    bd = torch.tensor(b, device=DEV)
    other = torch.cuda.Stream()
    with _solver(sys) as s:
        assert s.lsqr_one_launch()
        s.lsqr_solve(bd, 12, 0.0, 0.0)
        for _ in range(2):
            with torch.cuda.stream(other):
                torch.cuda._sleep(int(2.4e9))
                done = torch.cuda.Event()
                done.record()
            time.sleep(0.01)
            x, se, res = s.lsqr_solve(bd, 12, 0.0, 0.0)
            assert not done.query(), "the solve waited for the other stream"
            assert res["itn"] == ref["itn"]
            assert np.linalg.norm(x.cpu().numpy() - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])
            np.testing.assert_allclose(se.cpu().numpy(), ref["se"], rtol=1e-9)
            assert s.kernel_status() == _lib.GSR_OK
            other.synchronize()
        x2, _, _ = s.lsqr_solve(bd, 12, 0.0, 0.0)  # by the loop again
    assert np.linalg.norm(x2.cpu().numpy() - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])


def test_blocks_that_are_not_all_resident():
    # the loop leaves at its first barrier and the solve runs as launches
    sys = _random(257, 20, 37, 11, seed=9)
    b = oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4)
    ref = oracle.pc_lsqr(sys, b, 12, 0.0, 0.0)
    with _solver(sys) as s:
        assert s.lsqr_one_launch()
        for where in (2, 2, 0):
            s.inject_missing_block(where)
            for host in (False, True):
                for _ in range(2):
                    x, se, res = s.lsqr_solve(b if host else torch.tensor(b, device=DEV), 12, 0.0, 0.0)
                    x, se = (x, se) if host else (x.cpu().numpy(), se.cpu().numpy())
                    assert res["itn"] == ref["itn"]
                    assert np.linalg.norm(x - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])
                    np.testing.assert_allclose(se, ref["se"], rtol=1e-9)
                    assert s.kernel_status() == _lib.GSR_OK


def test_two_handles_from_two_threads():
    systems = [_random(257, 20, 37, 11, seed=9), _random(301, 25, 60, 30, seed=10)]
    refs, bs = [], []
    for sys in systems:
        bs.append(oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4))
        refs.append(oracle.pc_lsqr(sys, bs[-1], 12, 0.0, 0.0)["x"])
    errors = []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), _solver(systems[i]) as s:
                bd = torch.tensor(bs[i], device=DEV)
                for _ in range(30):
                    x, _, _ = s.lsqr_solve(bd, 12, 0.0, 0.0)
                    e = np.linalg.norm(x.cpu().numpy() - refs[i]) / np.linalg.norm(refs[i])
                    if not e <= 1e-9:
                        errors.append((i, e))
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
