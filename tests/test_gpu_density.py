"""Site density matrices in TF32 at chi = 32 and 64: through the fused chain kernel
where the graph has degree-3 sites (kernels="auto"), through the tile kernel
otherwise, both against the oracle at the same messages.

Tolerance: <Z> is a ratio of sums of products with six operands rounded to TF32
(the site tensor twice, three messages, one intermediate), each to 2^-11 at worst:
6 * 2^-11 = 3e-3.
"""
import numpy as np
import pytest

from oracle import bptn as OB
from oracle import graph as OG
from workloads import random_state

pytestmark = pytest.mark.gpu

GRAPHS = {
    "star": (7, [(0, 1), (0, 3), (0, 5), (1, 2), (3, 4), (5, 6)]),  # degrees 1, 2, 3
    "k4": (4, [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]),    # degree 3 alone
    "tee": (4, [(0, 1), (0, 2), (0, 3)]),                           # no degree 2
    "ring": (4, [(0, 1), (1, 2), (2, 3), (0, 3)]),                  # no degree 3
}


@pytest.fixture(scope="module")
def tnlib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_14887_gb300 import build
    build.build()
    import paper_2306_14887_gb300 as tn
    return tn


@pytest.mark.parametrize("chi", [32, 64])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_density_matches_oracle(tnlib, name, chi):
    n, edges = GRAPHS[name]
    g = OG.Graph(n, edges, OG.greedy_colouring(n, edges))
    tensors, msgs = random_state([g.degree(v) for v in range(n)], g.edges, chi, seed=chi)
    for kern in ("auto", "tile"):
        with tnlib.TNState(n, g.edges, g.colours, chi=chi, prec="tf32", kernels=kern) as s:
            for v in range(n):
                s.set_site(v, tensors[v])
            for (src, e), m in msgs.items():
                s.set_message(e, src, m)
            z = s.expect_z_all()
        o = OB.BPState(g, chi)
        o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
        o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
        assert np.abs(z - o.all_z()).max() < 3e-3, (name, kern)
