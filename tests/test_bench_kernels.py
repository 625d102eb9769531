"""The kernels that the benchmark's roofline names, their phases and their FP64 operations."""
import os
import re

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_2508_13986_gb300", "csrc")


def _source(*names):
    return "\n".join(open(os.path.join(CSRC, n)).read() for n in names)


@pytest.mark.parametrize("prec,macro", [("f64", "64"), ("f32", "32")])
def test_a_phase_names_the_kernels_that_it_brackets(prec, macro):
    """The lists of update_inst.cu (pre: grow, halo; post) in the order that the library
    launches and brackets them."""
    text = re.sub(r"//.*", "", _source("update_inst.cu"))
    body = text[text.index("void GBEES_ENTRY"):]
    head, tail = body.split("#if GBEES_PREC == 64")
    wide, narrow = tail.split("#else")
    lists = head + (wide if macro == "64" else narrow.split("#endif")[0])
    got = dict(re.findall(r"k->((?:pre|post)\[\d\]) = \(void\*\)(k_\w+)<", lists))
    k = bench.STEP_KERNELS[prec]
    assert k["grow"] == (got["pre[0]"], got["pre[1]"])
    assert k["faces"] == (got["post[0]"], got["post[1]"])
    assert k["apply"] == tuple(v for s, v in got.items() if s == "post[2]")


def test_every_kernel_exists_and_the_fp64_update_has_its_operations():
    text = _source("gbees_kernels.cuh")
    for prec, phases in bench.STEP_KERNELS.items():
        assert set(phases) == set(bench.BRACKETS)
        for name in sum(phases.values(), ()):
            assert re.search(rf"__global__ void [^;{{]*\b{name}\(", text), name
    for name in bench.STEP_KERNELS["f64"]["faces"] + bench.STEP_KERNELS["f64"]["apply"]:
        assert bench.fp64_flops_per_update(name, 6) > 0
