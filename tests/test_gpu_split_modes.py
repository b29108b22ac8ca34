"""The split-precision modes (TF32X3, BF16X3)."""
import numpy as np
import pytest

from oracle import graph as OG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnlib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_14887_gb300 import build
    build.build()
    import paper_2306_14887_gb300 as tn
    return tn


@pytest.mark.parametrize("solve", ["auto", "shared"])
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
def test_fp32_products_stop_as_fp32(tnlib, prec, solve):
    """kernels="auto" runs the products of FP32, so an evolution, which the stop rule and
    the solve's tolerance enter, is FP32's bit for bit."""
    g = OG.falcon27_patch()
    out = {}
    for p in ("fp32", prec):
        with tnlib.TNState(g.n, g.edges, g.colours, chi=8, prec=p, solve=solve) as s:
            s.apply_floquet(0.8, 6)
            out[p] = (s.stats()["bp_iters_total"], s.expect_z_all())
    assert out[prec][0] == out["fp32"][0]
    assert np.array_equal(out[prec][1], out["fp32"][1])
