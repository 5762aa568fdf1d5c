"""Rules of the bounded mbarrier waits, read off the sources: a time-out is not provoked in kernels that hold
tensor memory or have copies in flight.

* In a loop that contains warp-collective instructions the wait is the warp's, mbar_wait_warp: with
  mbar_wait the lanes decide one by one, and after a time-out those that stay would run
  collectives without those that left.
* Every mbarrier that copies or MMA completions arrive on is waited for once more, with a limit,
  before the CTA leaves (mbar_try_wait): nothing may land in its shared memory afterwards."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01522_gb300", "csrc")
COLLECTIVE = re.compile(r"tmem_ld\d|tmem_zero|__shfl|__syncwarp|__all_sync|__any_sync|__ballot_sync|mbar_wait_warp|\.sync\.aligned")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def enclosing_loop(text, pos):
    """Body of the innermost for / while loop around pos, '' where there is none."""
    depth = 0
    for i in range(pos, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth:
                depth -= 1
                continue
            head = text[max(0, i - 200):i].rstrip()
            head = head[max(head.rfind(c) for c in "{}") + 1:]
            if re.search(r"\b(for|while)\s*\([^{}]*\)$", head):
                d, j = 1, i + 1
                while d:
                    d += {"{": 1, "}": -1}.get(text[j], 0)
                    j += 1
                return text[i:j]
    return ""


@pytest.mark.parametrize("name", ["convnet.cu", "gemm_tcgen05.cu", "dense.cu"])
def test_waits_beside_warp_collectives_are_the_warps(name):
    text = source(name)
    calls = [m.start() for m in re.finditer(r"\bmbar_wait\(", text)]
    warp_calls = re.findall(r"\bmbar_wait_warp\(", text)
    assert calls or warp_calls
    for pos in calls:
        body = enclosing_loop(text, pos)
        assert not COLLECTIVE.search(body), f"{name}: per-lane wait in a loop with warp collectives:\n{body[:400]}"


@pytest.mark.parametrize("name", ["convnet.cu", "gemm_tcgen05.cu"])
def test_barriers_of_asynchronous_arrivals_are_drained(name):
    text = source(name)
    arriving = set(re.findall(r"\bmma_commit\(&(\w+)", text))
    for call in re.findall(r"\b(?:tma_load_\dd|bulk_load)\(([^;]*);", text):
        arriving |= set(re.findall(r"&(\w+)", call))
    barriers = set()
    for decl in re.findall(r"__shared__ __align__\(8\) uint64_t ([^;]*);", text):
        barriers |= set(re.findall(r"(\w+)(?:\[[^\]]*\])?(?:,|$)", decl))
    arriving &= barriers
    assert len(arriving) >= 3
    drained = set(re.findall(r"\bmbar_try_wait\(&(\w+)", text))
    assert arriving <= drained, f"{name}: not drained: {sorted(arriving - drained)}"
