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


@pytest.mark.parametrize("k", [3, 4])
def test_every_volume_variant_is_reported(k):
    g = _mk(4, k, 0)
    seen = set()
    for v in range(7):
        try:
            g.set_volume_variant(v)
        except Exception:
            g.clear_error()
            continue
        seen.add(v)
        assert g.tuning_volume()["variant"] == v
        assert g.tuning()["volume"] == ("tc" if v in (3, 6) else "fma")
    assert 6 in seen and 1 in seen


@pytest.mark.parametrize("k", [3, 4])
def test_every_timed_variant_has_a_time(k):
    """The autotuner of an FP32_TC context times variant 6, and keeps the fastest of those it reports."""
    t = _mk(10, k, 0).tuning_volume()
    assert t["ms"]["tensor_rows"] > 0
    names = ["reg_fused", "reg_split", "warp_fused", "tensor", "reg_tables_split", "reg_half_split", "tensor_rows"]
    assert names[t["variant"]] == min(t["ms"], key=t["ms"].get)


def test_times_of_the_c_call():
    import ctypes
    g = _mk(4, 4, 0)
    ms = (ctypes.c_double * 9)()
    assert g.lib.hopu_tuning_volume_ms(g.ctx, ms, 9) == 0
    assert list(ms[7:]) == [-1.0, -1.0] and ms[6] > 0 and ms[3] == -1.0
    assert g.lib.hopu_tuning_volume_ms(g.ctx, None, 9) != 0 and g.lib.hopu_tuning_volume_ms(None, ms, 9) != 0
    assert g.lib.hopu_tuning_volume_ms(g.ctx, ms, -1) != 0


def test_projection_at_k1():
    """The autotuner keeps the FMA projection at k = 1 in FP32_TC; tile_hint 2 still forces the other."""
    assert _mk(12, 1, 0).tuning()["v2l"] == "fma"
    assert _mk(12, 1, 2).tuning()["v2l"] == "tc"
