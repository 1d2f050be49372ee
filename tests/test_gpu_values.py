"""gsr_set_values: every copy of a replaced nonzero follows, so that the
products in all their forms and the solves belong to the new matrix."""
import numpy as np
import pytest

import oracle
from paper_2212_11675_gb300 import _lib, gen
from tests.test_gpu_forms import _abs, _random

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def _solver(sys, **kw):
    from paper_2212_11675_gb300.solver import Solver
    return Solver(sys, **kw)


def _replaced(sys, planes, seed):
    rng = np.random.default_rng(seed)
    v = sys.values.copy()
    for k in planes:
        v[:, k] = rng.standard_normal(sys.m)
    return gen.GaiaSystem(sys.n_stars, sys.n_dfa, sys.n_instr, sys.star_ptr, sys.attoff, sys.instr, v)


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


# 6,144 instruments are the limit of the row windows; in "repeated" a row names
# an instrument up to six times (slots of one row side by side in the sorted copy)
@pytest.mark.parametrize("n_instr,repeated", [(60, False), (9, True), (6144, False), (6145, False)])
@pytest.mark.parametrize("planes", [(17,), (22,), (0, 5, 16, 18, 20, 23)])
def test_products_after_replacing_planes(n_instr, repeated, planes):
    sys = _random(300, 12, 50, n_instr, seed=3)
    rng = np.random.default_rng(11)
    if repeated:
        sys.instr[:] = rng.integers(0, n_instr, size=sys.instr.shape)
        sys.instr[::7] = sys.instr[::7, :1]
    new = _replaced(sys, planes, 12)
    a = _abs(new)
    x, y = rng.standard_normal(sys.n), rng.standard_normal(sys.m)
    b1 = 1e-12 * oracle.aprod1(a, np.abs(x)) + 1e-300
    b2 = 1e-12 * oracle.aprod2(a, np.abs(y)) + 1e-300
    r1, r2 = oracle.aprod1_f32(new, x), oracle.aprod2_f32(new, y)
    for precision in (_lib.GSR_PREC_FP64, _lib.GSR_PREC_MIXED):
        with _solver(sys, precision=precision, conlim=0.0) as s:
            for k in planes:
                s.set_values(k, _dev(new.values[:, k]))
            forms = [(s.aprod1, s.aprod2, oracle.aprod1(new, x), oracle.aprod2(new, y))]
            if precision == _lib.GSR_PREC_MIXED:
                forms.append((s.aprod1_f32, s.aprod2_f32, r1, r2))
            for f1, f2, e1, e2 in forms:
                yd = torch.zeros(sys.m, dtype=torch.float64, device=DEV)
                xd = torch.zeros(sys.n, dtype=torch.float64, device=DEV)
                assert np.all(np.abs(f1(_dev(x), yd).cpu().numpy() - e1) <= b1), f1
                assert np.all(np.abs(f2(_dev(y), xd).cpu().numpy() - e2) <= b2), f2
            if precision == _lib.GSR_PREC_MIXED:
                Q, T = s.batched_products(_dev(x[None]), _dev(y[None]))
                # Q is stored in binary32: half an ulp on top
                h = 0.5 * np.spacing(np.abs(r1).astype(np.float32)).astype(np.float64)
                assert np.all(np.abs(Q.cpu().numpy()[0] - r1) <= b1 + h)
                assert np.all(np.abs(T.cpu().numpy()[0] - r2) <= b2)


def test_solves_after_replacing_an_instrument_plane():
    sys = _random(257, 20, 37, 11, seed=9)
    new = _replaced(sys, (17, 21), 13)
    b = oracle.aprod1(new, gen.x_true(new, 3)) + gen.noise(new, 4)
    ref = oracle.pc_lsqr(new, b, 5000, 1e-14, 1e-14, conlim=1e12)["x"]
    with _solver(sys, precision=_lib.GSR_PREC_MIXED, conlim=0.0) as s:
        for k in (17, 21):
            s.set_values(k, new.values[:, k].copy())  # from the host
        xs = [s.lsqr_solve(_dev(b), 5000, 1e-14, 1e-14)[0], s.mixed_solve(_dev(b), 20, 300, 1e-5, 1e-13)[0],
              s.batched_solve(_dev(b[None]), 20, 300, 1e-5, 1e-13)[0][0]]
    for x in xs:
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)


def test_norm_of_the_scaled_matrix_after_emptying_a_plane():
    # anorm^2 is the number of nonempty columns: zeros in plane 0 empty one
    # column a star, in plane 23 the global one
    sys = _random(40, 12, 10, 9, seed=3)
    b = np.random.default_rng(5).standard_normal(sys.m)
    with _solver(sys, precision=_lib.GSR_PREC_MIXED, conlim=0.0) as s:
        for planes, empty in (((), 0), ((0,), 40), ((23,), 41)):
            for k in planes:
                s.set_values(k, np.zeros(sys.m))
            for res in (s.mixed_solve(_dev(b), 1, 1)[1], s.batched_solve(_dev(b[None]), 1, 1)[1][0]):
                assert res["anorm"] == np.sqrt(sys.n - empty)
        s.set_values(0, sys.values[:, 0].copy())
        assert s.mixed_solve(_dev(b), 1, 1)[1]["anorm"] == np.sqrt(sys.n - 1)
