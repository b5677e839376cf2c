"""The autotuner's choice is made for the columns that a pass works on: runs of one size whose
truncations keep different shares of the columns (77 % and 35 %) do not share a cached choice, runs with
the same share do, and the choice of either leaves the results within FP32 rounding of the untuned ones."""
import json

import numpy as np
import pytest

from paper_2603_08892_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_choice_is_kept_per_share_of_columns(ns, monkeypatch, tmp_path):
    N = 128
    u = inputs.random_solenoidal(N, 17, kcut=N / 3, energy_total=1.0)
    cache = tmp_path / "tune.json"

    def run(kmax):
        with ns.Solver(N, 0.001, kmax, precision=ns.FP32, seed=3) as s:
            s.set_velocity(u)
            s.step(0.005, 2)
            return s.get_state()

    entries = []
    for kmax in (N / 2, N / 3, N / 2 - 0.25):
        monkeypatch.setenv("NS_AUTOTUNE_CACHE", str(cache))
        monkeypatch.delenv("NS_AUTOTUNE", raising=False)
        got = run(kmax)
        entries.append(len(json.loads(cache.read_text())))
        monkeypatch.setenv("NS_AUTOTUNE", "0")
        ref = run(kmax)
        assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref)
    assert entries == [1, 2, 2]
