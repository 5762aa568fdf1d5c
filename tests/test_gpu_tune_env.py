"""The knobs' environment variables are what a new context reports, with the values that they allow."""
import pytest

from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,lanes,want", [("384", "8", (384, 8)), ("512", "16", (512, 16)), ("100", "4", (256, 16))])
def test_environment_knobs_are_reported(monkeypatch, threads, lanes, want):
    need_gpu()
    monkeypatch.setenv("RSX_PASS2_THREADS", threads)
    monkeypatch.setenv("RSX_PASS2_LANES", lanes)
    t = rsx.Context((16, 16, 16), 0.4, "fp32").get_tuning()
    assert (t["p2_threads"], t["p2_lanes"]) == want
