"""The tuner finds the library's own defaults where they are the fastest, and does
not take a cached setting that was chosen without them (CPU; timing and the
device name are fakes)."""
import json

import pytest

pytest.importorskip("torch")


@pytest.fixture()
def at(monkeypatch):
    try:
        from paper_2208_12569_gb300 import autotune
    except (ImportError, OSError) as e:  # the library is built by __graft_entry__.build()
        pytest.skip("libfqsl.so not built: %s" % e)
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda *a: "FAKE GPU")
    return autotune


def _run(at, monkeypatch, calls):
    """A workload of few lines: fastest with the default chunk_tiles = 0."""
    current = {}

    def run_with(p):
        calls.append(p.chunk_tiles)
        current["p"] = p

    def cost(p):
        return 1.0 + (p.chunk_tiles != 0) + 0.01 * p.blocks_per_sm + 0.01 * p.sync_dirs + 0.001 * abs(p.refill_lanes - 32)

    monkeypatch.setattr(at, "_time", lambda run, reps: (run(), cost(current["p"]))[1])
    return run_with


def test_default_space_holds_the_defaults(at, monkeypatch):
    from paper_2208_12569_gb300 import fqsl

    best, _ = at.tune(_run(at, monkeypatch, []), fqsl.params(), key="w", path="")
    assert (best.chunk_tiles, best.blocks_per_sm, best.sync_dirs, best.refill_lanes) == (0, 0, 0, 32)


def test_setting_cached_without_them_is_tuned_again(at, monkeypatch, tmp_path):
    from paper_2208_12569_gb300 import fqsl

    path = str(tmp_path / "tune.json")
    calls = []
    run_with = _run(at, monkeypatch, calls)
    old = dict(at.DEFAULT_SPACE, chunk_tiles=(1, 4))
    best, _ = at.tune(run_with, fqsl.params(), key="w", path=path, space=old)
    assert best.chunk_tiles == 1
    best, table = at.tune(run_with, fqsl.params(), key="w", path=path)
    assert best.chunk_tiles == 0 and any(row["chunk_tiles"] == 0 for row in table)
    assert json.load(open(path))["FAKE GPU|w"]["best"]["chunk_tiles"] == 0
    calls.clear()
    again, _ = at.tune(run_with, fqsl.params(), key="w", path=path)
    # a search of part of the space is covered by the larger one
    part, _ = at.tune(run_with, fqsl.params(), key="w", path=path, space=old)
    assert calls == [] and again.chunk_tiles == part.chunk_tiles == 0
