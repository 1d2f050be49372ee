"""The dispatch rules at their edges: widths and remainders of the batched
columns, units and windows of the binary32 form, unit sizes and lane groups of
the FP64 aprod 2, the number of instruments that the staged aprod 1 takes, and
the one-launch LSQR loop beside the launched one.  Operators agree with the
oracle's same products within 1e-12 of sum |products|; solves within 1e-9."""
import numpy as np
import pytest

import oracle
from paper_2212_11675_gb300 import _lib, gen
from tests._dense import small

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def _solver(sys, **kw):
    from paper_2212_11675_gb300.solver import Solver
    return Solver(sys, **kw)


def _abs(sys):
    return gen.GaiaSystem(sys.n_stars, sys.n_dfa, sys.n_instr, sys.star_ptr, sys.attoff,
                          sys.instr, np.abs(sys.values))


def _random(S, rows, D, I, seed, offsets=None):
    """S stars of `rows` rows each; offsets uniform, or in runs drawn from `offsets`."""
    rng = np.random.default_rng(seed)
    m = S * rows
    sp = (np.arange(S + 1) * rows).astype(np.uint32)
    off = rng.integers(0, D - 3, size=m) if offsets is None else rng.choice(offsets, size=m)
    instr = np.argsort(rng.random((m, I)), axis=1)[:, :6] if I < 64 else \
        (rng.integers(0, I, size=(m, 1)) + np.arange(6) * (I // 6)) % I
    return gen.GaiaSystem(S, D, I, sp, off.astype(np.uint32), instr.astype(np.uint16),
                          rng.standard_normal((m, 24)))


def _vectors(sys, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(sys.n), rng.standard_normal(sys.m),
            rng.standard_normal(sys.m), rng.standard_normal(sys.n))


# (stars, rows per star, knots, instruments, offsets)
SHAPES = {
    "one_row": (1, 1, 4, 6, None),
    "tile_31": (31, 1, 5, 6, None),
    "tile_33": (3, 11, 5, 7, [1]),          # one offset, a tile and a row
    "one_offset": (700, 33, 9, 12, [3]),    # every unit in one segment
    "few_offsets": (900, 40, 7, 12, None),  # 4 offsets, many units each
    "many_offsets": (50, 40, 3000, 40, None),  # segments of 0, 1 and 2 rows
    "rows_127": (40, 127, 60, 30, None),    # lane groups of 8, 16 and 32
    "rows_129": (40, 129, 60, 30, None),
    "rows_257": (40, 257, 60, 30, None),
    "instr_3073": (300, 12, 50, 3073, None),
    "instr_6144": (300, 12, 50, 6144, None),
    "instr_6145": (300, 12, 50, 6145, None),
    "instr_6576": (300, 12, 50, 6576, None),  # the staged aprod 1's last
    "instr_6577": (300, 12, 50, 6577, None),
    "instr_6598": (300, 12, 50, 6598, None),
    "instr_6599": (300, 12, 50, 6599, None),
    "instr_12288": (300, 12, 50, 12288, None),  # the binary32 main pass's limits
    "instr_12289": (300, 12, 50, 12289, None),
    "instr_27648": (300, 12, 50, 27648, None),
    "instr_27649": (300, 12, 50, 27649, None),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_operators_at_edges(name):
    sys = _random(*SHAPES[name][:4], seed=3, offsets=SHAPES[name][4])
    x, y, y0, x0 = _vectors(sys, 4)
    a = _abs(sys)
    b1 = 1e-12 * (oracle.aprod1(a, np.abs(x)) + np.abs(y0)) + 1e-300
    b2 = 1e-12 * (oracle.aprod2(a, np.abs(y)) + np.abs(x0)) + 1e-300
    forms = [("aprod1", "aprod2", oracle.aprod1(sys, x, y0), oracle.aprod2(sys, y, x0)),
             ("aprod1_f32", "aprod2_f32", oracle.aprod1_f32(sys, x, y0),
              oracle.aprod2_f32(sys, y, x0))]
    with _solver(sys, precision=_lib.GSR_PREC_MIXED) as s:
        for f1, f2, r1, r2 in forms:
            for _ in range(2):  # counters and tickets are left as they were found
                yd, xd = torch.tensor(y0, device=DEV), torch.tensor(x0, device=DEV)
                getattr(s, f1)(torch.tensor(x, device=DEV), yd)
                getattr(s, f2)(torch.tensor(y, device=DEV), xd)
                e1 = np.max(np.abs(yd.cpu().numpy() - r1) / b1)
                e2 = np.max(np.abs(xd.cpu().numpy() - r2) / b2)
                assert e1 <= 1.0 and e2 <= 1.0, (f1, e1, e2)
        assert s.kernel_status() == _lib.GSR_OK


def test_staged_after_a_smaller_handle():
    # the launch attribute of the staged kernels is per function, not per
    # handle; 6,576 instruments fill the 227 KB that a block may have: 16 bytes
    # each in steps of 128, beside 18 stages of 7,048 bytes and 256 static bytes
    big = _random(300, 12, 50, 6576, seed=5)
    x, _, y0, _ = _vectors(big, 6)
    b1 = 1e-12 * (oracle.aprod1(_abs(big), np.abs(x)) + np.abs(y0)) + 1e-300
    with _solver(big) as s, _solver(gen.make("tiny")) as t:
        assert s.aprod1_staging() and t.aprod1_staging()
        yd = torch.tensor(y0, device=DEV)
        s.aprod1(torch.tensor(x, device=DEV), yd)
        assert np.all(np.abs(yd.cpu().numpy() - oracle.aprod1(big, x, y0)) <= b1)


@pytest.mark.parametrize("k,kt,lanes", [(1, 8, 8), (2, 8, 16), (6, 4, 32), (7, 2, 8), (9, 8, 8),
                                        (13, 4, 16), (19, 8, 32)])
def test_batched_columns(k, kt, lanes):
    sys = _random(*SHAPES["few_offsets"][:4], seed=7)
    rng = np.random.default_rng(k)
    X, Y = rng.standard_normal((k, sys.n)), rng.standard_normal((k, sys.m))
    a = _abs(sys)
    with _solver(sys, precision=_lib.GSR_PREC_MIXED, conlim=0.0) as s:
        s.set_batch_tiling(kt, lanes)
        Q, T = s.batched_products(torch.tensor(X, device=DEV), torch.tensor(Y, device=DEV))
        Q, T = Q.cpu().numpy(), T.cpu().numpy()
    for c in range(k):
        r1, r2 = oracle.aprod1_f32(sys, X[c]), oracle.aprod2_f32(sys, Y[c])
        # Q is stored in binary32: half an ulp on top of the accumulation bound
        h = 0.5 * np.spacing(np.abs(r1).astype(np.float32)).astype(np.float64)
        assert np.all(np.abs(Q[c] - r1) <= 1e-12 * oracle.aprod1(a, np.abs(X[c])) + h), c
        assert np.all(np.abs(T[c] - r2) <= 1e-12 * oracle.aprod2(a, np.abs(Y[c]))), c


@pytest.mark.parametrize("S,k", [(257, 9), (257, 17)])
def test_batched_solve_two_runs(S, k):
    # two runs of columns side by side, columns that stop at different iterations
    sys = small(S, 37, 11, seed=31)
    ax = oracle.aprod1(sys, gen.x_true(sys, 3))
    B = np.stack([ax * 10.0 ** -j + gen.noise(sys, 100 + j) for j in range(k)])
    with _solver(sys, precision=_lib.GSR_PREC_MIXED, conlim=0.0) as s:
        X, res = s.batched_solve(torch.tensor(B, device=DEV), max_outer=20, max_inner=300,
                                 inner_tol=1e-5, atol=1e-13)
        X = X.cpu().numpy()
    for j in range(k):
        ref = oracle.pc_lsqr(sys, B[j], 5000, 1e-14, 1e-14, conlim=1e12)
        assert res[j]["converged"] == 1, (j, res[j])
        assert np.linalg.norm(X[j] - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"]), j


# the one-launch loop takes systems of at most 400,000 rows
@pytest.mark.parametrize("shape", [(40, 1, 8, 7), (257, 20, 37, 11), (1000, 400, 60, 30),
                                   (1000, 401, 60, 30)])
@pytest.mark.parametrize("itmax", [1, 12])
def test_lsqr_loop_and_launches(shape, itmax):
    sys = _random(*shape, seed=9)
    b = oracle.aprod1(sys, gen.x_true(sys, 3)) + gen.noise(sys, 4)
    ref = oracle.pc_lsqr(sys, b, itmax, 0.0, 0.0)
    with _solver(sys) as s:
        for _ in range(2):
            x, se, res = s.lsqr_solve(torch.tensor(b, device=DEV), itmax, 0.0, 0.0)
            assert res["itn"] == ref["itn"] == itmax
            x = x.cpu().numpy()
            assert np.linalg.norm(x - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])
            for key in ("rnorm", "anorm", "xnorm"):
                assert res[key] == pytest.approx(ref[key], rel=1e-9), key
            np.testing.assert_allclose(se.cpu().numpy(), ref["se"], rtol=1e-9)
        assert s.kernel_status() == _lib.GSR_OK
