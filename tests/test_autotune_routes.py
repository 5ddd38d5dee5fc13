"""The autotuner beside the resident solves: nothing is searched for a batch whose
instances all run resident, only the others' classes in a mixed one, and entries written
before the route existed are not used."""
import json

import pytest

from paper_2408_03452_gb300 import autotune

SMALL, LARGE = (48, 48, 24), (256, 256, 256)


@pytest.fixture
def fake(monkeypatch):
    calls = []

    def cost(grids, zc, coef, coef64, b, tol, maxit, precond, sweep=0, tile=0):
        calls.append((list(zc), sweep, tile))
        return 1.0 + abs(zc[-1] - 32) + sweep + tile

    monkeypatch.setattr(autotune, "_time_batch", cost)
    monkeypatch.setattr(autotune, "_resident", lambda grids, coef: [tuple(g) == SMALL for g in grids])
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda *a: "fake-device")
    return calls


def test_resident_batch_is_not_searched(fake):
    r = autotune.tune_batch([SMALL] * 3, None, None, None)
    assert len(fake) == 1 and (r["sweep"], r["tile"]) == (0, 0) and r["zc"] == [4] * 3


def test_mixed_batch_searches_the_classes_in_the_sweeps(fake):
    r = autotune.tune_batch([SMALL, LARGE], None, None, None)
    assert r["zc"][1] == 32 and (r["sweep"], r["tile"]) == (0, 0)
    # the common run, the kernels, then two trials for the one class
    assert len(fake) == len(autotune.CANDIDATES) + 4 + 2


def test_older_entries_miss(fake, tmp_path):
    cache = str(tmp_path / "zc.json")
    autotune.tune_batch([SMALL], None, None, None, cache=cache)
    db = json.load(open(cache))
    (key,) = db
    old = json.dumps(json.loads(key)[:-1])
    json.dump({old: {"zc": [[list(SMALL), 128]], "sweep": 1, "tile": 2, "ms_per_solve": 9.0}},
              open(cache, "w"))
    r = autotune.tune_batch([SMALL], None, None, None, cache=cache)
    assert (r["sweep"], r["tile"], r["zc"]) == (0, 0, [4]) and r["ms_per_solve"] != 9.0
