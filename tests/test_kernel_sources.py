"""Orders inside the CUDA kernels that no run can show to be kept: read from the sources.

A kernel that allocates TMEM lets its successors start (programmatic dependent launch) only after
the allocation.  The other way round a successor's CTA can take the columns of an SM first and then
wait for the kernel whose CTA waits for those columns.

A warp that only issues MMAs waits for the previous kernel before its first bounded wait for the
workers, as the workers do, and follows the limit of hopu_set_wait_limit upwards: otherwise a long
predecessor, or a raised limit, would make it give up work that was never late.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_06698_gb300", "csrc")


def kernels(word):
    """(file, text) of every __global__ function whose body holds `word`, comments removed."""
    out = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cuh", ".cu")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            out += [(name, part) for part in re.split(r"(?=__global__)", text)[1:] if word in part]
    return out


TMEM = kernels("tmem_alloc(")


def test_tmem_kernels_are_found():
    assert len(TMEM) >= 5


@pytest.mark.parametrize("i", range(len(TMEM)))
def test_dependents_start_after_the_tmem_allocation(i):
    name, body = TMEM[i]
    alloc, trigger = body.index("tmem_alloc("), body.index("pdl_trigger()")
    assert trigger > alloc, name
    # the same warp, in order: nothing but the end of the statement between the two
    assert re.fullmatch(r"tmem_alloc\(tslot, C::TCOLS\);\s*pdl_trigger\(\)", body[alloc:trigger + len("pdl_trigger()")]), name
    assert body.count("pdl_trigger()") == 1, name


MMA_WARP = kernels("warp == NT / 32")


def test_mma_warp_kernels_are_found():
    assert len(MMA_WARP) >= 2


@pytest.mark.parametrize("i", range(len(MMA_WARP)))
def test_mma_warp_waits(i):
    name, body = MMA_WARP[i]
    body = body[body.index("warp == NT / 32"):]
    body = body[:body.index("} else {")]                # the MMA warp's branch
    assert body.index("pdl_wait()") < body.index("mbar_wait("), name
    assert "mma_warp_limit(m.tc_wait_limit)" in body, name
    # the waits for the workers take that limit; only the final drain keeps the default
    assert len(re.findall(r"mbar_wait\([^;]*, limit\)", body)) == 2, name
    assert "1u << 24" not in body, name


def members(struct):
    """Names of the data members of a struct of hopu_internal.h."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "hopu_internal.h")).read())
    body = text[text.index(f"struct {struct} {{"):]
    body = body[:body.index("};")]
    return re.findall(r"\b(\w+)\s*=", body)


@pytest.mark.parametrize("struct,var", [("DevMesh", "m"), ("DevTabs", "tb")])
def test_every_array_of_a_context_is_read(struct, var):
    """What every launch copies as an argument is read by a kernel (or named at a launch)."""
    text = "".join(re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, n)).read()) for n in sorted(os.listdir(CSRC))
                   if n.endswith(".cuh"))
    capi = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "capi.cu")).read())
    names = members(struct)
    assert len(names) >= 8
    for name in names:
        read = re.search(rf"\b{var}\.{name}\b", text) or re.search(rf"c->dm\.{name}\b(?!\s*=[^=])", capi)
        assert read, f"{struct}::{name}"
