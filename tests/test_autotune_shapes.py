"""The autotuner's search (CPU only, no timing): every candidate is another launch of the sweep, the defaults cover
threads per SM between 256 and the maximum, and a grid with equal launches times each once."""
import pytest

from paper_1608_04601_gb300 import autotune as A
from paper_1608_04601_gb300 import workloads as W
from paper_1608_04601_gb300 import xsections as X


def _launch(block, ppt, ctas, precision):
    """(chunk, threads) of the sweep's launch by the options' definition in the C header."""
    top = 768 if precision == "fp32" else 512
    return 32 * (4 if block == 512 and ppt == 8 else ppt), min(top, block * ctas) if ctas else top


def _timed(monkeypatch, tmp_path, precision, **kw):
    calls = []

    def time_config(gases, discharges, precision, block, ppt, ctas, sort_every, steps=12, warmup=4):
        calls.append(_launch(block, ppt, ctas, precision) + (sort_every,))
        return float(len(calls))

    monkeypatch.setattr(A, "time_config", time_config)
    monkeypatch.setattr(A, "_key", lambda *a: "k")
    monkeypatch.setattr(A, "CACHE", str(tmp_path / "cache.json"))
    best = A.autotune(X.he_like(eps_max_eV=50.0, de_eV=1.0), W.c1(), precision, use_cache=False, **kw)
    assert best["searched"] == len(calls) and best["ms_per_step"] == 1.0
    return calls


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_default_candidates_differ(monkeypatch, tmp_path, precision):
    calls = _timed(monkeypatch, tmp_path, precision)
    assert len(set(calls)) == len(calls)
    threads = {t for _, t, _ in calls}
    assert {c for c, _, _ in calls} == {64, 128, 256} and {256, max(threads)} <= threads
    assert precision == "fp64" or any(256 < t < 768 for t in threads)


def test_equal_launches_are_timed_once(monkeypatch, tmp_path):
    calls = _timed(monkeypatch, tmp_path, "fp32", tiles=[(256, 4), (128, 4), (512, 8), (256, 8)], ctas=[0, 2], sorts=[8])
    assert sorted(calls) == [(128, 256, 8), (128, 512, 8), (128, 768, 8), (256, 512, 8), (256, 768, 8)]
