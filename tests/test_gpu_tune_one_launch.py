"""Split counts and the sweep that runs as one launch (FP32, chi <= 32): the counts
belong to the plan's separate launches, so neither tuning nor a table changes what
such a handle computes, bit for bit."""
import numpy as np
import pytest

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


def sweep(s, g, tensors, msgs):
    for v in range(g.n):
        s.set_site(v, tensors[v])
    for (src, e), m in msgs.items():
        s.set_message(e, src, m)
    s.bp_converge(tol=1e30, max_iters=1)
    return {k: s.get_message(k[1], k[0]) for k in msgs}


@pytest.mark.parametrize("chi", [16, 23])
def test_tuning_and_tables_leave_the_messages(tnlib, chi):
    g = OG.eagle127()
    tensors, msgs = random_state([g.degree(v) for v in range(g.n)], g.edges, chi, seed=chi)
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi) as s:
        plain = sweep(s, g, tensors, msgs)
        tuned = sweep(s, g, tensors, msgs) if s.autotune(reps=2) else None
    assert all(np.array_equal(plain[k], tuned[k]) for k in msgs)
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi) as s:
        rows = [ln.split() for ln in s.autotune(reps=1).splitlines()]
    # the same table without a split
    assert any(r[7] != "1" for r in rows)
    table = "".join(" ".join(r[:7] + ["1", r[8]]) + "\n" for r in rows)
    with tnlib.TNState(g.n, g.edges, g.colours, chi=chi) as s:
        s.apply_tuning(table)
        given = sweep(s, g, tensors, msgs)
    assert all(np.array_equal(plain[k], given[k]) for k in msgs)
