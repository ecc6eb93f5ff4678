"""The tests of test_gpu_pairs.py on rows that are not 16-byte aligned, which the warp
strips alone take, two iterations per launch (k_binary_strip2): certificates in the last
pair's launch, the solve loop device-driven and host-driven, schedules.  (On aligned
rows the same calls run the chains of warps.)"""
import pytest

from test_gpu_pairs import *  # noqa: F401,F403 (its tests and fixtures)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def unaligned_rows(cmf, monkeypatch):  # noqa: F811
    monkeypatch.setattr(cmf, "pitch_for", lambda w: (w + 3) // 4 * 4 + 2)
