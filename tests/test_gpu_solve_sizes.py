"""The refined truncation solve at sizes between the powers of two: tile and
warp remainders, the switch between the solve's Jacobi orders, and both sides of
the switch to the cluster kernels at chi = 64.

Tolerance as for the powers of two: the spectrum equals the exact FP64 spectrum
of the solve's own FP32-rounded Gram inputs to 1e-11."""
import numpy as np
import pytest

from test_gpu_solve import gram_exact_spectrum, make_case, run_solve, tnlib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [1, 2, 5, 17, 24, 33, 47, 48, 49, 63, 80, 96, 112, 144])
def test_refined_spectrum_between_powers_of_two(tnlib, chi):  # noqa: F811
    n_edges = 3
    _, gram = make_case(chi, 2 * chi + 3, n_edges, seed=chi, decay=5.0 / chi)
    _, s = run_solve(tnlib, gram, chi, 1 if chi % 2 else -1, n_edges, "refined")
    for k in range(n_edges):
        ref = gram_exact_spectrum(gram[k], chi, 1 if chi % 2 else -1)
        assert np.abs(s[k] - ref).max() < 1e-11
