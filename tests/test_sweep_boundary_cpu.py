"""Order of memory in the sweeps' cooperative launch, read in the source (a
missing order need not show in any run): a block's wait at a level boundary
acquires what the other blocks' arrivals released, before the barrier that
lets its threads go on, and what other blocks write within the launch is read
by coherent loads that the compiler keeps behind that wait."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
with open(os.path.join(ROOT, "paper_2406_07441_gb300", "csrc", "lskum_kernels.cu")) as f:
    SRC = re.sub(r"//[^\n]*", "", f.read())


def _body(name):
    """The definition of a function: from its name to the brace at the line's start that closes it."""
    m = re.search(r"\b%s\([^;{]*\)\s*\n\{(.*?)\n\}" % name, SRC, re.S)
    assert m, name
    return m.group(1)


def test_the_wait_acquires_between_the_poll_and_the_barrier():
    assert re.search(r"__syncthreads\(\);.*red\.release\.gpu", _body("boundary_arrive"), re.S)
    wait = _body("boundary_wait")
    assert re.search(r"(ld\.acquire\.gpu|fence\.acq_rel\.gpu|__threadfence\(\)).*__syncthreads\(\)", wait, re.S)


def test_what_other_blocks_write_is_not_read_as_read_only_data():
    loads = re.findall(r"load4?_l2\(const (?:double|float) \*p[^{]*\)\n\{(.*?)\n\}", SRC, re.S)
    assert len(loads) >= 2
    for body in loads:  # volatile, with a memory clobber, not through the read-only path
        assert "asm volatile" in body and '"memory"' in body and ".nc" not in body and "__ldg" not in body
    # the increments, the axis products and (formed in the launch's first step)
    # the framed points' Jacobians
    for name in ("lane_load", "sweep_interior", "framed_load", "framed_run", "sweep_framed", "sweep_point"):
        for call in re.findall(r"\b(load4|__ldcg|__ldg)\(([^,;]*)", _body(name)):
            what = call[1].strip()
            assert re.match(r"d\.(g0|pk_g0)\b", what), (name, call)  # (of an earlier launch)
