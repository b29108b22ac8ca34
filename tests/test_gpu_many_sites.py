"""More than 16383 sites of one degree: the leg transposes of such a handle (TF32,
chi = 32, with degree-3 sites) need more than one launch's blocks."""
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


def test_density_matrices_of_a_long_chain(tnlib):
    """A path of 16400 degree-2 sites hung on a star, in |0..0> but for three sites turned
    by theta: <Z> is one, and cos(theta) there to the TF32 rounding of a density matrix's
    two tensors and two messages (4 * 2^-11)."""
    n = 16404
    edges = [(0, 1), (0, 2), (0, 3)] + [(i, i + 1) for i in range(3, n - 1)]
    theta = 0.5
    with tnlib.TNState(n, edges, OG.greedy_colouring(n, edges), chi=32, prec="tf32") as s:
        assert np.array_equal(s.expect_z_all(), np.ones(n))
        t = np.zeros((2, 32, 32), np.complex64)
        t[:, 0, 0] = np.cos(theta / 2), -1j * np.sin(theta / 2)
        for v in (4, 16385, n - 2):
            s.set_site(v, t)
        z = s.expect_z_all()
        for v in (4, 16385, n - 2):
            assert abs(z[v] - np.cos(theta)) < 2e-3
        assert z[5] == 1.0 and z[16384] == 1.0
