"""Rules of the kernels' sources that a run cannot show: a fault against one
of them needs a device wait to run out at a particular moment, or another
compiler's choice of a load."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_09421_gb300", "csrc")


def _sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def test_a_cta_leaves_a_timed_out_march_as_one():
    """No thread returns on its own read of the timeout word: the kernels'
    barriers count threads that would have left."""
    for name, text in _sources().items():
        assert not re.search(r"\*\s*static_cast<(const )?volatile int\s*\*>\(a\.err\)\)\s*\{?\s*return", text), name


def test_dependent_launches_read_the_launch_before_by_plain_loads():
    """A pass that is alive while the pass before it writes (u for an x-pass, R
    for a y-pass) takes no read-only pointer
    to it, and loads it by cp.async or plain loads behind its wait."""
    text = _sources()["rte_kernels.cu"]
    for kernel, what in (("xpass_kernel", "U"), ("ypass_kernel", "R")):
        at = text.index(kernel + "(StepArgs")
        signature = text[at:text.index("{", at)]
        assert re.search(r"const float\*\s+%s\b" % what, signature), (kernel, signature)
    y = text[text.index("ypass_kernel(StepArgs"):text.index("fluence_kernel(")]
    assert "ld_plain4(R +" in y and not re.search(r"(ld4|__ldg)\(R \+", y)
    assert y.index("griddepcontrol.wait;") < y.index("ld_plain4(R +")
    # the one-tile tensor-core x-pass: no C++ load of u
    body = _sources()["rte_tc.cu"]
    body = body[body.index("void tc_pass_body("):body.index("tc_pass_kernel(StepArgs")]
    assert not re.search(r"reinterpret_cast<const float4\*>\(U \+", body)


def test_a_dependent_launch_waits_before_it_leaves():
    """A one-tile pass ends after the launch it depends on, also where it
    does no work: the march clears the timeout word after its last launch."""
    text = _sources()["rte_tc.cu"]
    body = text[text.index("void tc_pass_body("):text.index("main loop over K chunks")]
    exits = [m.start() for m in re.finditer(r"\breturn;", body)]
    assert len(exits) == 2                     # the timeout word, the injected expiry
    for at in exits:
        assert "griddepcontrol.wait;" in body[at - 120:at]
