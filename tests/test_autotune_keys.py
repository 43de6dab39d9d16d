"""What the tile autotuner's cache is keyed by, without a GPU: the threads that
the batch's CTAs run (the sample has to run as many), the form of the class's
blocks and the library's sources."""
import numpy as np
import pytest

from paper_1807_00370_gb300 import autotune


@pytest.fixture
def tuner(monkeypatch, tmp_path):
    calls = []

    def fake(mt, m, k, device=None, n_blocks=512, verbose=False, threads=256):
        calls.append((mt, m, threads))
        return (len(calls), 1, 8), {}

    monkeypatch.setattr(autotune, "tune_class", fake)
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "tiles.json"))
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda d: "GPU")
    return calls


def test_cache_key(tuner, monkeypatch):
    dev = object()
    first = autotune.tiles_for([8], [4], dev, threads=256)
    assert autotune.tiles_for([8], [4], dev, threads=256) == first and len(tuner) == 1
    assert autotune.tiles_for([8], [4], dev, threads=512) != first
    assert tuner[-1] == (8, 8, 512)
    assert autotune.tiles_for([5], [4], dev, threads=256) != first      # FMA form of the class
    monkeypatch.setattr(autotune._build, "source_hash", lambda: "other")
    assert autotune.tiles_for([8], [4], dev, threads=256) != first
    assert len(tuner) == 4


def test_threads_of_batch_and_sample():
    one = np.ones(1)
    assert autotune.batch_threads(100 * one, 8 * one, 4 * one, 152) == 512
    # the samples of tune_class
    for threads, n in ((256, 4 * 152), (512, 2 * 152 - 1)):
        e = np.ones(n)
        assert autotune.batch_threads(512 * e, 8 * e, 4 * e, 152) == threads
