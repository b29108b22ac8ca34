"""The CUDA-core FP32 GEMM at the edges of its tiles and slices: one BP sweep of
a degree-3 star (its mode products, rows- and column-contiguous outputs, and the
split-K closes) against the FP64 oracle's sweep.

Tolerance: the messages have unit Frobenius norm, and each goes through two mode
products and a close.  Every sum is taken in 16-deep complex slices, 32 FP32
products each, whose worst-case relative error is 32 * 2^-24 = 1.9e-6; the slice
sums are added error-free.  Three stages: 6e-6.
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


def one_sweep(tn, g, chi, tensors, msgs, prec):
    with tn.TNState(g.n, g.edges, g.colours, chi=chi, prec=prec) as s:
        for v in range(g.n):
            s.set_site(v, tensors[v])
        for (src, e), m in msgs.items():
            s.set_message(e, src, m)
        s.bp_converge(tol=1e30, max_iters=1)
        return {k: s.get_message(k[1], k[0]) for k in msgs}, s.expect_z_all()


@pytest.mark.parametrize("chi", [1, 2, 3, 8, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 96])
def test_sweep_matches_oracle(tnlib, chi):
    g = OG.star3_tree()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=chi)
    got, z = one_sweep(tnlib, g, chi, tensors, msgs, "fp32")
    o = OB.BPState(g, chi)
    o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
    o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
    o.bp_sweep()
    assert max(float(np.linalg.norm(got[k] - o.M[k])) for k in o.M) < 6e-6
    # the split modes run their contractions in the same kernel
    for prec in ("tf32x3", "bf16x3"):
        same, z2 = one_sweep(tnlib, g, chi, tensors, msgs, prec)
        assert all(np.array_equal(same[k], got[k]) for k in got) and np.array_equal(z, z2)


@pytest.mark.parametrize("chi", [1, 2, 3, 7, 8, 9, 13, 16])
def test_small_chi_sweep_in_a_union(tnlib, chi):
    """At chi <= 16 a sweep's contractions run as one launch over (site, open leg,
    open-leg block) jobs: every message is the same bit for bit alone and as one
    of three components."""
    g = OG.star3_tree()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=100 + chi)
    alone, _ = one_sweep(tnlib, g, chi, tensors, msgs, "fp32")
    n, e, c, offs = tnlib.batch_union([(g.n, g.edges, g.colours)] * 3)
    with tnlib.TNState(n, e, c, chi=chi) as s:
        for off in offs:
            for v in range(g.n):
                s.set_site(off + v, tensors[v])
        for i, off in enumerate(offs):
            for (src, ed), m in msgs.items():
                s.set_message(i * len(g.edges) + ed, off + src, m)
        s.bp_converge(tol=1e30, max_iters=1)
        for i, off in enumerate(offs):
            for src, ed in msgs:
                got = s.get_message(i * len(g.edges) + ed, off + src)
                assert np.array_equal(got, alone[(src, ed)])


@pytest.mark.parametrize("chi", [17, 18, 19, 20, 21, 22, 23, 24, 25])
def test_streamed_sweep(tnlib, chi):
    """At chi = 17 .. 24 a CTA holds the slabs of a block of open-leg values and
    streams the site tensor for the close (25: back to GEMM launches): against the
    oracle, and the same bit for bit as one of two components.  Tolerance as above."""
    g = OG.star3_tree()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=300 + chi)
    alone, _ = one_sweep(tnlib, g, chi, tensors, msgs, "fp32")
    o = OB.BPState(g, chi)
    o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
    o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
    o.bp_sweep()
    assert max(float(np.linalg.norm(alone[k] - o.M[k])) for k in o.M) < 6e-6
    n, e, c, offs = tnlib.batch_union([(g.n, g.edges, g.colours)] * 2)
    with tnlib.TNState(n, e, c, chi=chi) as s:
        for i, off in enumerate(offs):
            for v in range(g.n):
                s.set_site(off + v, tensors[v])
            for (src, ed), m in msgs.items():
                s.set_message(i * len(g.edges) + ed, off + src, m)
        s.bp_converge(tol=1e30, max_iters=1)
        if chi <= 24:
            for i, off in enumerate(offs):
                for src, ed in msgs:
                    got = s.get_message(i * len(g.edges) + ed, off + src)
                    assert np.array_equal(got, alone[(src, ed)])


@pytest.mark.parametrize("chi", [25, 26, 27, 28, 29, 30, 31, 32])
def test_wide_streamed_sweep(tnlib, chi):
    """chi = 25 .. 32, two warps to a slab: against the oracle, as one of two
    components bit for bit the same, and as one of 52 (over four CTAs per SM, where
    multiples of four run as GEMM launches) against the oracle again.  Tolerance as
    above."""
    g = OG.star3_tree()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=400 + chi)
    alone, _ = one_sweep(tnlib, g, chi, tensors, msgs, "fp32")
    o = OB.BPState(g, chi)
    o.T = [t.astype(np.complex64).astype(complex) for t in tensors]
    o.M = {k: m.astype(np.complex64).astype(complex) for k, m in msgs.items()}
    o.bp_sweep()
    assert max(float(np.linalg.norm(alone[k] - o.M[k])) for k in o.M) < 6e-6
    for copies in (2, 52):
        n, e, c, offs = tnlib.batch_union([(g.n, g.edges, g.colours)] * copies)
        with tnlib.TNState(n, e, c, chi=chi) as s:
            for i, off in enumerate(offs):
                for v in range(g.n):
                    s.set_site(off + v, tensors[v])
                for (src, ed), m in msgs.items():
                    s.set_message(i * len(g.edges) + ed, off + src, m)
            s.bp_converge(tol=1e30, max_iters=1)
            for i in (0, copies - 1):
                for src, ed in msgs:
                    got = s.get_message(i * len(g.edges) + ed, offs[i] + src)
                    assert float(np.linalg.norm(got - o.M[(src, ed)])) < 6e-6
                    if copies == 2:
                        assert np.array_equal(got, alone[(src, ed)])


@pytest.mark.parametrize("chi", [4, 5, 7, 8, 9, 13, 15, 16, 17])
def test_one_launch_environments(tnlib, chi):
    """Up to chi = 16 a gate layer's environments run as one launch (17: GEMM
    launches): four steps on the star, where bond dimension 4 is exact, against the
    oracle, within the FP32 path's 1e-6 for exact evolutions.  Sites of degree 1, 2
    and 3, every leg open."""
    g = OG.star3_tree()
    o = OB.run(g, chi, 0.6, 4)
    for prec in ("fp32", "tf32x3"):
        with tnlib.TNState(g.n, g.edges, g.colours, chi=chi, prec=prec) as s:
            s.apply_floquet(0.6, 4)
            assert np.abs(s.expect_z_all() - o.all_z()).max() < 1e-6


@pytest.mark.parametrize("chi", [18, 21, 23, 24, 25, 27, 28, 31, 32, 33])
def test_streamed_environments(tnlib, chi):
    """The environments of chi = 17 .. 32 through the streamed sweep kernels, one part
    per physical value: as above, same bound."""
    g = OG.star3_tree()
    o = OB.run(g, 8, 0.6, 4)  # bond dimension 4 is exact
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi) as s:
        s.apply_floquet(0.6, 4)
        assert np.abs(s.expect_z_all() - o.all_z()).max() < 1e-6
