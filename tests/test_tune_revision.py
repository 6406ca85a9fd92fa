"""Picks cached for other launch shapes are not applied: the key of a batch holds
the revision of the detection kernel and of what a tuning means (host code)."""
import numpy as np
import pytest

# the key of this batch before keys held a revision
OLD_KEY = ("gpu=NVIDIA GB300|sm=152|p=9,13|k=1|q=3|b=19|rule=0|lo=0"
           "|jobs=1241x376:L8:s3f99999a:e20:c32:f2000:m11")


@pytest.fixture(scope="module")
def binding():
    from paper_2410_04090_gb300 import build
    build.build()
    from paper_2410_04090_gb300 import jslam
    return jslam


def test_entries_without_a_revision_miss(binding, tmp_path):
    img = np.zeros((376, 1241), np.uint8)
    key = binding.tune_key("NVIDIA GB300", 152, {}, [binding.Job(img, img)])
    assert [f for f in key.split("|") if not f.startswith("rev=")] == OLD_KEY.split("|")  # the same batch
    path = str(tmp_path / "tune.json")
    binding.tune_cache_put(path, OLD_KEY, (64, 64, 0, 2, 0), 0.5)
    assert binding.tune_cache_get(path, key) is None
    binding.tune_cache_put(path, key, (128, 64, 0, 0, 0), 0.4)  # beside the old entry
    assert binding.tune_cache_get(path, key) == (128, 64, 0, 0, 0)
    assert binding.tune_cache_get(path, OLD_KEY) == (64, 64, 0, 2, 0)
