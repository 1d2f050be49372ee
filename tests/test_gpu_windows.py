"""Row windows of the binary32 instrument pass that do not fit: every window
uses other instruments heavily, so a block's sums exceed its shared memory and
the instrument-sorted copy serves instead."""
import pytest

from paper_2212_11675_gb300 import _lib, gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def test_sums_beyond_shared_memory_use_the_sorted_copy():
    from paper_2212_11675_gb300.solver import Solver
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    # 14 windows of 8,160 rows a block, six instruments in each: 14 x 6 x 204
    # columns of 40 entries, above the 16,384 sums of a block
    W, rounds, lam = 8160, 14, 80
    m = W * nsm * rounds
    S, D = m // lam, 50000
    g = torch.Generator(device=DEV).manual_seed(3)
    row = torch.arange(m, device=DEV)
    ins = (6 * (row // (W * nsm)))[:, None] + torch.arange(6, device=DEV)
    att = torch.randint(0, D - 3, (m,), generator=g, device=DEV)
    values = torch.randn((m, 24), generator=g, dtype=torch.float64, device=DEV)
    ptr = torch.arange(S + 1, device=DEV) * lam
    y = torch.randn(m, generator=g, dtype=torch.float64, device=DEV)
    # the instrument columns of A32^T y and the sum of their |terms|
    t = (values[:, 17:23].float() * y.float()[:, None]).double()
    ref = torch.zeros(6 * rounds, dtype=torch.float64, device=DEV)
    ref.index_add_(0, ins.reshape(-1), t.reshape(-1))
    scale = torch.zeros_like(ref).index_add_(0, ins.reshape(-1), t.abs().reshape(-1))
    del t
    held = {}
    for n_instr in (6144, 6145):  # beyond 6,144 there are no row windows
        sys = gen.GaiaSystem(S, D, n_instr, ptr.to(torch.uint32), att.to(torch.uint32),
                             ins.to(torch.uint16), values)
        torch.cuda.synchronize()
        with Solver(sys, precision=_lib.GSR_PREC_MIXED) as s:
            held[n_instr] = s.device_bytes
            for _ in range(2):
                x = s.aprod2_f32(y, torch.zeros(s.n, dtype=torch.float64, device=DEV))
                q = x[5 * S + 3 * D:-1]
                assert torch.all((q[:6 * rounds] - ref).abs() <= 1e-12 * scale)
                assert not q[6 * rounds:].any()
            assert s.kernel_status() == _lib.GSR_OK
    # no row windows are kept that no pass reads (36 bytes a row)
    assert held[6144] <= held[6145] + m
