"""Kernels launched with programmatic dependent launch (launch_after) run while their predecessor still writes. CUDA's
read-only loads (__ldg, and what the compiler makes of const __restrict__ parameters) are defined only for data that nobody
writes during the kernel, so these kernels may use them for the geometry alone. Checked on the sources: a violation need
not show in results."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_12891_gb300", "csrc")
SOURCES = {f: open(os.path.join(CSRC, f)).read() for f in ("dg_kernels.cuh", "dg_fixed.cuh", "dg_fixed_lift.cuh")}
TEXT = "\n".join(SOURCES.values())
# device functions that these kernels hand the chain's arrays to, with the parameter
HELPERS = [("load_state", "U"), ("wall_face", "U"), ("lift_node", "Wse"), ("fx_viscous", "Fn")]


def _parameters(name):
    m = re.search(r"\b%s\(((?:const|int)[^{;]*)\)\s*\{" % name, TEXT)
    assert m, name
    return [p.strip() for p in m.group(1).split(",")]


def test_the_dependently_launched_kernels():
    assert set(re.findall(r"launch_after\((k_\w+)", TEXT)) == {"k_face", "k_lift_fx", "k_volume_fx"}


@pytest.mark.parametrize("kernel", ["k_face", "k_lift_fx", "k_volume_fx"])
def test_no_restrict_on_read_parameters(kernel):
    bad = [p for p in _parameters(kernel) if "__restrict__" in p and p.startswith("const")]
    assert not bad, bad


@pytest.mark.parametrize("helper,name", HELPERS)
def test_no_restrict_in_helpers(helper, name):
    (p,) = [p for p in _parameters(helper) if re.search(r"\b%s$" % name, p)]
    assert "__restrict__" not in p, p


@pytest.mark.parametrize("source", ["dg_fixed.cuh", "dg_fixed_lift.cuh"])
def test_read_only_loads_are_of_metric_terms(source):
    for m in re.finditer(r"__ldg\((\w+)", SOURCES[source]):
        assert m.group(1) in ("Je", "Jd"), m.group(0)  # (element's Ja)


@pytest.mark.parametrize("kernel", ["k_face", "k_lift_fx", "k_volume_fx"])
def test_waits_before_reading(kernel):
    """The kernel waits for its predecessor, and lets its successor start only after that."""
    body = TEXT[re.search(r"\b%s\(const DgDevice d" % kernel, TEXT).end():]
    wait, nxt = body.find("wait_for_previous();"), body.find("let_next_start();")
    assert 0 <= wait < nxt < (body.find("__global__") % len(body))
    assert "load_state" not in body[:wait]
