"""The FP32 sweep and gate environments up to chi = 32 in both forms: as one launch
each, and as the plan's separate launches of the CUDA-core GEMM.

Up to chi = 16 the two take every sum in the same order: the same bits.  The separate
launches are held to the oracle at every size, odd ones above all (4-byte copies,
partial tiles and slices): the messages have unit norm, and each goes through two mode
products and a close, every sum in 16-deep slices of 32 FP32 products, 32 * 2^-24 =
1.9e-6 apiece: 6e-6.
"""
import numpy as np
import pytest

from oracle import bptn as OB
from oracle import graph as OG
from workloads import random_state

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


def loaded(tn, g, chi, tensors, msgs, separate):
    s = tn.TNState(g.n, g.edges, g.colours, chi=chi)
    if separate:
        assert tn.lib().tnbp_separate_launches(s._h) == 0
    for v in range(g.n):
        s.set_site(v, tensors[v])
    for (src, e), m in msgs.items():
        s.set_message(e, src, m)
    return s


@pytest.mark.parametrize("graph", [OG.star3_tree(), OG.falcon27_patch()], ids=["star7", "patch27"])
@pytest.mark.parametrize("chi", [1, 2, 3, 5, 7, 8, 9, 13, 15, 16])
def test_both_forms_give_the_same_bits(tnlib, graph, chi):
    g = graph
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=600 + chi)
    out, launches = [], []
    for separate in (False, True):
        with loaded(tnlib, g, chi, tensors, msgs, separate) as s:
            s.apply_floquet(0.7, 1, check=False)
            launches.append(s.stats()["kernel_launches"])
            out.append([s.get_site(v) for v in range(g.n)] +
                       [s.get_message(e, src) for src, e in msgs] +
                       [s.bond_spectrum(e) for e in range(len(g.edges))])
    assert launches[0] < launches[1]
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("chi", [1, 2, 3, 7, 8, 15, 16, 17, 18, 23, 24, 25, 28, 31, 32])
def test_separate_launches_match_the_oracle(tnlib, chi):
    g = OG.star3_tree()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=700 + chi)
    o = OB.BPState(g, chi)
    o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
    o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
    o.bp_sweep()
    with loaded(tnlib, g, chi, tensors, msgs, True) as s:
        s.bp_converge(tol=1e30, max_iters=1)
        for src, e in msgs:
            assert float(np.linalg.norm(s.get_message(e, src) - o.M[(src, e)])) < 6e-6
