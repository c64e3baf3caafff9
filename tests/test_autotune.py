"""The launch-shape autotuner's choice among its candidates, on made-up times."""
import json

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def tuner(gbaes, monkeypatch, tmp_path):
    """autotune with a cache of its own; tuner.times: ms by shape (1.0 where absent)."""
    from paper_1201_0398_gb300 import autotune

    monkeypatch.setenv("GBAES_TUNE_CACHE", str(tmp_path / "tune_cache.json"))
    shapes = iter(())

    def fake(fn, reps, stream):
        nonlocal shapes
        fn()
        shape = next(shapes, None)
        if shape is None:
            shapes = iter(autotune.ECB_CANDIDATES)
            shape = next(shapes)
        return autotune.times.get(shape, 1.0)

    monkeypatch.setattr(autotune, "_time", fake)
    monkeypatch.setattr(autotune, "times", {}, raising=False)
    yield autotune
    gbaes.set_tuning(128, False, 0, 0)


@pytest.mark.gpu
def test_the_shape_by_size_stays_unless_another_is_faster(gbaes, tuner):
    tuner.times[1024, 2] = 0.995
    hit = tuner.tune_ecb(128, False, nbytes=1 << 16)
    assert (hit["threads"], hit["blocks_per_thread"]) == gbaes.tuning(128, False) == (0, 0)
    tuner.times[1024, 2] = 0.9
    hit = tuner.tune_ecb(128, False, nbytes=1 << 16, force=True)
    assert (hit["threads"], hit["blocks_per_thread"]) == gbaes.tuning(128, False) == (1024, 2)
    tuner.times[512, 4] = 0.8
    hit = tuner.tune_ecb(128, False, nbytes=1 << 16, force=True, apply=False)
    assert (hit["threads"], hit["blocks_per_thread"]) == (512, 4) and gbaes.tuning(128, False) == (1024, 2)


@pytest.mark.gpu
def test_shapes_of_another_kernel_are_not_used(gbaes, tuner):
    """Entries of a cache file written by other kernel sources, or before it named them."""
    tuner.times[1024, 2] = 0.9
    first = tuner.tune_ecb(128, False, nbytes=1 << 16)
    assert tuner.tune_ecb(128, False, nbytes=1 << 16) == first  # (from the file)
    with open(tuner.cache_path()) as f:
        (key, hit), = json.load(f).items()
    name, kernel, rest = key.split("|", 1)[1].split("|", 2)
    for other in (f"ecb|{name}|{rest}", f"ecb|{name}|{'0' * len(kernel)}|{rest}"):
        with open(tuner.cache_path(), "w") as f:
            json.dump({other: dict(hit, threads=768, blocks_per_thread=4)}, f)
        got = tuner.tune_ecb(128, False, nbytes=1 << 16)
        assert (got["threads"], got["blocks_per_thread"]) == gbaes.tuning(128, False) == (1024, 2)
