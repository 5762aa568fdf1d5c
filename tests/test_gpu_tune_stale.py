"""Knobs that were good for other kernels do not stick: cache entries of an earlier version are not
applied, and a search that starts with the work plane in global scratch can leave it (64^3, where
shared memory holds the plane and is several times faster)."""
import pytest
import torch

from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tag", ["rsx2", "rsx3"])
def test_entries_of_earlier_versions_are_not_applied(tmp_path, tag):
    need_gpu()
    prop = torch.cuda.get_device_properties(0)
    cache = tmp_path / "tune.txt"
    cache.write_text(f"{tag} 24 24 24 fp32 3 5 {prop.multi_processor_count} {prop.name}|256 1 0 1 16 0.1000\n")
    ctx = rsx.Context((24, 24, 24), 0.35, "fp32")
    t = ctx.autotune(3, 5, cache=str(cache))
    assert t["best_ms"] > 0 and t["p2_global"] == 0
    again = rsx.Context((24, 24, 24), 0.35, "fp32").autotune(3, 5, cache=str(cache))
    assert again["best_ms"] == -1.0 and again["chunk_outputs"] == t["chunk_outputs"]


def test_the_search_leaves_the_global_plane():
    need_gpu()
    ctx = rsx.Context((64, 64, 64), 0.25, "fp32")
    ctx.set_tuning(p2_global=1)
    assert ctx.autotune(8, 16)["p2_global"] == 0
