"""The passes that may be launched while the kernel before them still runs (programmatic stream
serialisation) do not read what that kernel writes as data that is constant for the whole kernel: no
ld.global.nc, that is no __ldg and no const __restrict__ pointer, for the orbitals and the
intermediate.  Read off the sources: the race itself depends on the compiler's scheduling."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01522_gb300", "csrc")
KERNELS = [("poisson_xpass.cuh", "k_pass1"), ("poisson_pass2.cuh", "k_pass2"), ("poisson_xpass.cuh", "k_pass3")]
# tables written once, with a device synchronisation, when a context is created
CONSTANT = {"twx", "twg", "vl"}
TABLE_READS = {"vsrc"}   # k_pass2: a row of vl


def kernel(fname, name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fname)).read())
    start = re.search(rf"\b{name}\(Geom", text).start()
    args, body = text[start:].split("{", 1)
    end = body.find("__global__")
    return args, body[:end if end > 0 else None]


@pytest.mark.parametrize("fname,name", KERNELS)
def test_dependent_data_is_read_coherently(fname, name):
    args, body = kernel(fname, name)
    assert "pdl_wait();" in body
    restricted = set(re.findall(r"__restrict__ (\w+)", args))
    assert restricted <= CONSTANT, f"{name}: __restrict__ on {sorted(restricted - CONSTANT)}"
    for call in re.findall(r"__ldg\(([^;]*)", body):
        assert any(re.search(rf"\b{t}\b", call) for t in TABLE_READS), f"{name}: __ldg({call}"
    head = body.split("pdl_wait();")[0]
    assert not re.search(r"\b(inter|f1|f2|pm)\b\s*[\[.+]", head), f"{name}: dependent data before the wait"


def test_every_kernel_launched_with_the_attribute_is_covered():
    launched = set()
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"launch_pdl\(g{1,2}\.pdl, k,", text):
            launched.add(re.findall(r"auto k = (?:k_)?(pass\d)", text[:m.start()])[-1])
    assert launched == {"pass1", "pass2", "pass3"}
