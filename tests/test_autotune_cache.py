"""The autotuner times every distinct launch once and keeps a timing only for the kernels it was taken
of (host only, no GPU)."""
import pytest

from paper_1006_2716_gb300 import autotune


@pytest.mark.parametrize("L", [8, 32, 40, 64])
def test_one_candidate_of_the_fixed_point_kernel(L):
    default = 1 if L <= 32 else 4
    assert [c for c in autotune.candidates(L, dtau_U=2.0) if c[0] == 0] == [(0, default, 1)]
    assert [c for c in autotune.candidates(L, dtau_U=3.0) if c[0] == 0] == [(0, default, 1)]
    wide = [c for c in autotune.candidates(L) if c[0] == 0]
    assert [c for c in autotune.candidates(L, dtau_U=3.5) if c[0] == 0] == wide and len(wide) > 1
    pairs = [c for c in autotune.candidates(L) if c[0] == 2]
    assert [c for c in autotune.candidates(L, dtau_U=2.0) if c[0] == 2] == pairs


def test_cached_timings_are_dropped_when_a_kernel_changes(tmp_path, monkeypatch):
    import torch

    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "gpu")
    monkeypatch.setattr(autotune, "_CACHE", str(tmp_path / "autotune.json"))
    calls = []

    def probe(L, chains, form, tw, k, *rest):
        calls.append((form, tw, k))
        return float(len(calls))

    monkeypatch.setattr(autotune, "_probe", probe)
    first = autotune.tune([32], 8, forms=(0,))
    assert calls == [(0, 1, 1)]
    assert autotune.tune([32], 8, forms=(0,)) == first and len(calls) == 1
    monkeypatch.setattr(autotune, "sources_digest", lambda: "changed")
    autotune.tune([32], 8, forms=(0,))
    assert len(calls) == 2
