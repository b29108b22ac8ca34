"""The split-precision modes (TF32X3, BF16X3) in both forms: as FP32 products on the
CUDA cores (kernels="auto") and as split products in the tensor-core tile kernel
(kernels="tile").

Bounds of the split products: hi*hi + hi*lo + lo*hi drops lo*lo, about 2^-22 (TF32X3)
and 2^-16 (BF16X3) relative, plus FP32 accumulation: 2e-6 and 5e-6 in a message of
unit norm after one sweep; 3e-5 and 1e-4 in <Z> of an evolution, which the residual
floor of the arithmetic adds to.
"""
import numpy as np
import pytest

from oracle import bptn as OB
from oracle import graph as OG
from workloads import random_state

pytestmark = pytest.mark.gpu

SWEEP_TOL = {"tf32x3": 2e-6, "bf16x3": 5e-6}
Z_TOL = {"tf32x3": 3e-5, "bf16x3": 1e-4}


@pytest.fixture(scope="module")
def tnlib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_14887_gb300 import build
    build.build()
    import paper_2306_14887_gb300 as tn
    return tn


# on 27 qubits a degree-3 launch has 262144 multiply-adds or more from chi = 16 on, so
# that the tile kernel takes it
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("graph,chi", [(OG.falcon27_patch(), 16), (OG.falcon27_patch(), 23),
                                       (OG.star3_tree(), 32), (OG.star3_tree(), 64)],
                         ids=["patch27-16", "patch27-23", "star7-32", "star7-64"])
def test_split_products_sweep(tnlib, prec, graph, chi):
    g = graph
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=11)
    got = {}
    for kern in ("auto", "tile"):
        with tnlib.TNState(g.n, g.edges, g.colours, chi=chi, prec=prec, kernels=kern) as s:
            for v in range(g.n):
                s.set_site(v, tensors[v])
            for (src, e), m in msgs.items():
                s.set_message(e, src, m)
            s.bp_converge(tol=1e30, max_iters=1)
            got[kern] = {k: s.get_message(k[1], k[0]) for k in msgs}
    o = OB.BPState(g, chi)
    o.T = [t.astype(complex) for t in tensors]
    o.M = {k: m.astype(complex) for k, m in msgs.items()}
    o.bp_sweep()
    for kern in got:
        assert max(np.abs(got[kern][k] - o.M[k]).max() for k in o.M) < SWEEP_TOL[prec], kern
    # two forms indeed
    assert any(not np.array_equal(got["auto"][k], got["tile"][k]) for k in msgs)


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("chi,steps", [(16, 4), (8, 6)], ids=["exact", "truncated"])
def test_split_products_evolution(tnlib, prec, chi, steps):
    g = OG.eagle127()
    o = OB.run(g, chi, 0.6, steps)
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi, prec=prec, kernels="tile") as s:
        s.apply_floquet(0.6, steps)
        assert np.abs(s.expect_z_all() - o.all_z()).max() < Z_TOL[prec]


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
