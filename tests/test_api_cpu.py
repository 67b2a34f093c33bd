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


def test_no_stream_means_the_current_one(api, monkeypatch):
    """None and any other false value; elsewhere the API writes `stream or the current one`."""
    import torch
    monkeypatch.setattr(api, "_current_raw_stream", lambda index: 40 + index)
    for none in (None, 0, False):
        assert api._raw_stream(none, torch.device("cuda", 2)) == 42

    class Stream:
        cuda_stream = 7

    assert api._raw_stream(Stream(), torch.device("cuda", 2)) == 7
