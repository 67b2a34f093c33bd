"""Argument handling of the torch-facing API that needs no GPU."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def api():
    pytest.importorskip("torch")
    from paper_1705_06661_gb300 import api
    return api


def test_coefficients_of_any_dimension(api):
    """A ready coefficient array is taken as it is, whatever d; d outside 2..4 is refused behind this
    (ValueError, or the library's own error), never by an IndexError."""
    for d, n in ((2, 2), (4, 24), (5, 120)):
        c = np.ones((2, n))
        assert api._coef_chain(c, d) is c
        with pytest.raises(ValueError):
            api._coef_chain(np.ones((2, n + 1)), d)
    with pytest.raises(ValueError):
        api._coef_chain(np.ones((1, 24)), -1)
