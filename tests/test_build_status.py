"""The build refuses a dropped status of the launch functions: a graph whose
loop body was captured short of the kernel that clears the loop flag would
instantiate and never end."""
import os
import subprocess

import pytest

from paper_2212_11675_gb300 import build

PROBE = """#include "gsr_internal.cuh"
cudaError_t probe(gsr_handle_t *h, cudaStream_t s)
{
    %s
    return cudaSuccess;
}
"""
CALLS = ["gsr::enqueue_iteration(h, s, 0, 1)", "gsr::build_cg_graph(h)", "gsr::run_batched_inner(h, 1, 1, s)"]


def _compile(tmp_path, body):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "probe.cu"
    src.write_text(PROBE % body)
    inc = ["-I", build.CSRC, "-I", os.path.join(os.path.dirname(build.HERE), "include")]
    return subprocess.run([cc, *build.ARCH, *build.FLAGS, *inc, "-c", str(src), "-o", os.devnull],
                          capture_output=True, text=True)


@pytest.mark.parametrize("call", CALLS)
def test_dropped_status_does_not_build(tmp_path, call):
    r = _compile(tmp_path, call + ";")
    assert r.returncode != 0 and "nodiscard" in r.stderr, r.stderr


def test_status_that_is_read_builds(tmp_path):
    r = _compile(tmp_path, "if (cudaError_t e = %s) return e;" % CALLS[0])
    assert r.returncode == 0, r.stderr
