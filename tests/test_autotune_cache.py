"""The tuning cache, without a GPU: a pick is found again with the library it was
made with, and not with another one."""
import pytest

from paper_1806_10889_gb300 import autotune
from paper_1806_10889_gb300.workloads import TissueSpec


class _Tuned(Exception):
    """Raised in the place of tuning."""


@pytest.fixture
def cache(tmp_path, monkeypatch):
    so = tmp_path / "libtissue.so"
    so.write_bytes(b"one")
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "_gpu_name", lambda: "gpu")
    monkeypatch.setattr(autotune, "lib", lambda: None)
    monkeypatch.setattr(autotune, "library_path", lambda: str(so))

    def tune(*a, **k):
        raise _Tuned
    monkeypatch.setattr(autotune, "Tissue", tune)
    monkeypatch.setattr(autotune, "tissue_candidates", lambda V: [(1, 16, 1, 0, 0)])
    return so


class _Member:
    def __init__(self, spec):
        self.spec = spec

    def read_counts(self):
        raise _Tuned


def test_a_pick_of_another_build_is_not_taken_over(cache):
    spec = TissueSpec(64, 64, 16, seed=1)
    members = [_Member(spec)]
    # as versions without the build in the key wrote it
    autotune._store("tissue|gpu|V=256|cells~4096|dt=0.1", {"config": [1, 16, 1, 0, 0], "ms": {}})
    autotune._store("batch|gpu|dt=0.1|256:4096", {"classes": {"256": [16, 1, 0]}, "steps_per_graph": 1})
    for content in (b"one", b"two"):
        cache.write_bytes(content)
        with pytest.raises(_Tuned):
            autotune.tune_tissue(spec, 0.1)
        with pytest.raises(_Tuned):
            autotune.tune_batch(members, 0.1)
    build = autotune._build()
    autotune._store(f"tissue|gpu|{build}|V=256|cells~4096|dt=0.1",
                    {"config": [1, 8, 2, 0, 1], "ms": {}})
    autotune._store(f"batch|gpu|{build}|dt=0.1|256:4096",
                    {"classes": {"256": [8, 2, 1]}, "steps_per_graph": 4})
    assert autotune.tune_tissue(spec, 0.1)["config"] == (1, 8, 2, 0, 1)
    assert autotune.tune_batch(members, 0.1)["classes"] == {256: (8, 2, 1)}
    cache.write_bytes(b"three")
    with pytest.raises(_Tuned):
        autotune.tune_tissue(spec, 0.1)
