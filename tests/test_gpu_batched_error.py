"""Accumulation error of the batched A^T Y, from exact sums of its binary32
products: as small as that of one row per lane with a tree over the lanes.
Bounds: twice the rms errors of the kernels' summation orders restated in
numpy (stars of 400 rows 6.4e-18, offsets of 200 rows 2.5e-18 of the sum of
|terms|, rounded up); chains over all rows of a slot or of a unit of eight
tiles have 2.9e-17 and 4.3e-17."""
import numpy as np
import pytest

from paper_2212_11675_gb300 import _lib
from tests._dense import columns
from tests.test_gpu_forms import _random

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _exact(cols, terms, n):
    order = np.argsort(cols, kind="stable")
    c, t = cols[order], terms[order].astype(np.longdouble)
    cut = np.flatnonzero(np.r_[True, c[1:] != c[:-1]])
    total, scale = np.zeros(n, np.longdouble), np.zeros(n, np.longdouble)
    total[c[cut]] = np.add.reduceat(t, cut)
    scale[c[cut]] = np.add.reduceat(np.abs(t), cut)
    return total, scale


def test_rms_error_of_star_and_attitude_sums():
    from paper_2212_11675_gb300.solver import Solver
    # 1.3e6 rows: units of eight tiles; 400 rows a star, 200 an offset
    sys = _random(3250, 400, 6503, 60, seed=21)
    rng = np.random.default_rng(22)
    Y = rng.standard_normal((8, sys.m))
    with Solver(sys, precision=_lib.GSR_PREC_MIXED) as s:
        s.set_batch_tiling(8, 16)
        _, T = s.batched_products(torch.zeros((8, sys.n), dtype=torch.float64, device="cuda"),
                                  torch.tensor(Y, device="cuda"))
        T = T.cpu().numpy()
    cols = columns(sys)
    for j in (0, 5):
        terms = sys.values.astype(np.float32) * Y[j].astype(np.float32)[:, None]
        for part, bound in ((slice(0, 5), 1.3e-17), (slice(5, 17), 6e-18)):
            total, scale = _exact(cols[:, part].ravel(), terms[:, part].ravel(), sys.n)
            used = scale > 0
            e = ((T[j] - total)[used] / scale[used]).astype(np.float64)
            assert np.sqrt(np.mean(e * e)) <= bound, (j, part, np.sqrt(np.mean(e * e)))
