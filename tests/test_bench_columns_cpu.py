"""The roofline of bench.py counts the bytes of the columns that the passes touch: those with a mode
inside the truncation, as the oracle's mask has them, and the byte model is scaled by their share."""
import inspect

import pytest

import bench
from oracle import spectral as sp


@pytest.mark.parametrize("N,kmax", [(16, 8.0), (24, 8.0), (32, 14.6), (48, 23.999)])
def test_share_of_columns(N, kmax):
    mask = sp.truncation_mask(N, kmax)  # [kz][ky][kx]
    assert bench.kept_columns(N, kmax) == mask.any(axis=0).sum() / (N * (N // 2))


def test_roofline_counts_no_skipped_column():
    src = inspect.getsource(bench)
    assert "14.0 * C * kept" in src and "8.0 * C * kept" in src
    assert src.count("model_bytes_per_step() * kept") == 2
