"""What hopu_tuning and hopu_tuning_volume report is the kernel that runs."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _mk(n, k, hint, prec="f32_tc"):
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(3, n)
    return Hopu(m.coords, m.elems, m.rep, k=k, l=k - 1, prec=prec, tile_hint=hint)


def test_tile_hint_2_does_not_depend_on_timing():
    """Variant 6 is the fastest at these sizes and is not what tile_hint 2 stands for."""
    assert _mk(10, 3, 2).tuning_volume()["variant"] == 3
    t = _mk(10, 4, 2).tuning_volume()
    assert t["variant"] in (0, 1, 4, 5) and "tensor_rows" not in t["ms"]
