"""Memory rules of the fused pass that no run can show reliably, checked in its source
(csrc/tl_pass_impl.cuh): a pass is launched while its predecessor, which writes
its inputs, may still run."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_2607_24908_gb300", "csrc", "tl_pass_impl.cuh")


def code():
    with open(SOURCE) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_read_only_loads_only_of_the_hosts_tables():
    """__ldg wants memory unmodified for the kernel's lifetime: of what a pass
    reads, only the item table of a batch is."""
    args = re.findall(r"__ldg\(([^)]*)\)", code())
    assert args and all(a.startswith("first_item") for a in args), args
    assert "ld.global.nc" not in code()


def test_the_last_tiles_lanes_are_ordered_after_the_ticket():
    """finish_tile: lane 0 takes the ticket, all lanes then read what other CTAs
    wrote. Between the two every lane passes a __syncwarp (a shuffle hands over the
    value but orders no memory) and a fence."""
    body = code().split("void finish_tile(", 1)[1].split("\n}\n", 1)[0]
    after = body[body.index("atomicAdd"):body.index("__ldcg(slots")]
    assert "__syncwarp()" in after and "__threadfence()" in after.split("__syncwarp()", 1)[1]
    assert after.index("__syncwarp()") < after.index("sc->a")
