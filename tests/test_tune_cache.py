"""Cached tuning choices made among earlier kernels are searched for again."""
import json
import types

import pytest

torch = pytest.importorskip("torch")


def test_choices_among_earlier_kernels_are_searched_again(tmp_path, monkeypatch):
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: types.SimpleNamespace(
        multi_processor_count=152, name="test device"))
    p = cmf.default_params(2, 4)
    problem = types.SimpleNamespace(H=64, W=64, L=4, params=p, u=torch.zeros(1))
    calls = []

    def search(s):
        calls.append(s)
        return cmf.default_params(2, 4, variant=8), 1.0

    monkeypatch.setattr(cmf, "cmf_autotune_potts", search)
    old = "|".join(str(v) for v in ("potts", 64, 64, 4, p.storage, p.algo, p.impl, p.tune_step,
                                    p.c, p.phase_storage, p.phase_gap, 152, "test device"))
    path = tmp_path / "tune.json"
    path.write_text(json.dumps({old: {"variant": 2, "sweeps": 1, "ms_to_gap": 1.0}}))
    for _ in range(2):  # the second time from the cache
        assert cmf.tuned_params(problem, cache_path=str(path)).variant == 8
    assert len(calls) == 1
    assert old in json.loads(path.read_text())  # other libraries' entries stay
