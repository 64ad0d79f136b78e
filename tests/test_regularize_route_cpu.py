"""Which form of the mesh regularisation a context gets: the 16-block cluster,
the portable 8-block one where that is refused, one block where both are, and
what is kept of an answer that could not be had.  No GPU needed."""
import ctypes

import pytest


@pytest.mark.parametrize("nodes", [1, 2562, 16384, 16385, 32768, 32769])
@pytest.mark.parametrize("fits16,fits8,widest,known", [
    (1, 1, 16, 1), (1, 0, 16, 1), (0, 1, 8, 1), (0, 0, 0, 1), (-1, 1, 8, 0), (-1, 0, 0, 0), (0, -1, 0, 0), (-1, -1, 0, 0)])
def test_cluster_of_a_context(nodes, fits16, fits8, widest, known):
    from paper_2403_01161_gb300 import _lib, build

    build.build()
    k = ctypes.c_int(-1)
    ctas = _lib.load().ibl_test_regularize_ctas(nodes, fits16, fits8, ctypes.byref(k))
    assert k.value == known
    assert ctas == (widest if nodes <= 2048 * widest else 0)
