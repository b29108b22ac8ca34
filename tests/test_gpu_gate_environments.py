"""Gate environments of a saturated random state, every leg open, against the oracle.

The bond spectra that a first gate layer leaves come straight from the environments of
its edges.  Tolerance: an environment G has an error of at most 6e-6 of its norm (two
mode products and a close, each a sum of 16-deep FP32 slices, 1.9e-6 apiece), that is
6e-6 cond(G) relative to G in its own metric, and the squared singular values of the
bond move by at most the sum of both sides' relative errors: half that sum for the
values themselves, with both condition numbers taken from the oracle.
"""
import numpy as np
import pytest

from oracle import bptn as OB
from oracle import graph as OG
from workloads import random_psd, random_site_tensor, rng

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


def saturated_state(g, chi, seed):
    """Random tensors of full rank whose environments are well conditioned: matrices near
    the identity on degree-2 sites, messages near the identity."""
    r = rng(seed)
    tensors = []
    for v in range(g.n):
        t = random_site_tensor(r, g.degree(v), [chi] * g.degree(v))
        tensors.append(np.eye(chi) + 0.2 / np.sqrt(chi) * t if g.degree(v) == 2 else t)
    msgs = {}
    for e, ends in enumerate(g.edges):
        for v in ends:
            m = np.eye(chi) / np.sqrt(chi) + 0.3 * random_psd(r, chi)
            msgs[(v, e)] = m / np.linalg.norm(m)
    return tensors, msgs


def first_layer(g, chi, tensors, msgs, theta):
    """{edge: (normalised singular values, relative tolerance)} of the first gate layer."""
    o = OB.BPState(g, chi)
    o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
    o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
    o.apply_rx(theta)
    out = {}
    for e in g.layers()[0]:
        v, w = g.edges[e]
        a, b = OB.gate_split(+1)
        xv = o._absorbed_matrix(v, e, a)[0]
        xw = o._absorbed_matrix(w, e, b)[0]
        rv, rw = np.linalg.qr(xv)[1], np.linalg.qr(xw)[1]
        s = np.linalg.svd(rv @ rw.T, compute_uv=False)[:chi]
        cond = np.linalg.cond(rv) ** 2 + np.linalg.cond(rw) ** 2
        out[e] = (s / np.linalg.norm(s), 0.5 * 6e-6 * cond)
    return out


@pytest.mark.parametrize("chi", [3, 8, 15, 16, 17, 19, 23, 24, 25, 27, 28, 31, 32, 33])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_first_layer_spectra(tnlib, chi, shift):
    tree = OG.star3_tree()
    g = OG.Graph(tree.n, tree.edges, [(c + shift) % 3 for c in tree.colours])
    tensors, msgs = saturated_state(g, chi, 500 + chi)
    want = first_layer(g, chi, tensors, msgs, 0.7)
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi) as s:
        for v in range(g.n):
            s.set_site(v, tensors[v])
        for (src, e), m in msgs.items():
            s.set_message(e, src, m)
        s.apply_floquet(0.7, 1, check=False)
        for e, (spec, tol) in want.items():
            assert tol < 1e-4
            # (a leaf's bond holds two values; what FP32 Gram matrices leave beyond
            # them, about 1e-4, is not compared)
            got = s.bond_spectrum(e)[:len(spec)]
            assert (np.abs(got - spec) <= tol * spec).all(), (e, tol)
