"""The register-resident FP32 kernels over every order, against the FP64 oracle.

Small meshes whose facet and element counts are no multiple of a warp's share, so that the
last group of every launch is ragged and element records start at every offset modulo 16
bytes; random data and per-facet orders; walls and inlets; a wind of its own and w = u.
Tolerance: the stated FP32 bound of the operator, 1e-6 of the largest output.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import adjoint as A
from oracle import convection as C
from oracle import fe, hdiv, mesh, rk

pytestmark = pytest.mark.gpu

ORDERS = [(2, 3, 1), (2, 5, 2), (2, 4, 3), (2, 3, 4), (3, 3, 1), (3, 4, 2), (3, 3, 3), (3, 3, 4), (3, 3, 5)]


def _rel(got, ref):
    got = got.detach().double().cpu().numpy().reshape(-1)
    return float(np.abs(got - np.asarray(ref).reshape(-1)).max() / np.abs(ref).max())


def _setup(dim, n, k, walls):
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(dim, n)
    rep = None if walls else m.rep
    g = Hopu(m.coords, m.elems, rep, k=k, l=k - 1, prec="f32")
    topo = mesh.MeshTopo(m.coords, m.elems, rep)
    return g, topo, fe.ref_element(dim, k)

# past one element per resident warp, where the separate-wind volume term changes kernels
LARGER = [(2, 41, 2), (3, 8, 2), (3, 9, 3), (3, 8, 4), (3, 6, 5)]


@pytest.mark.parametrize("dim,n,k", LARGER)
def test_separate_wind_volume_kernels(dim, n, k):
    g, topo, ref = _setup(dim, n, k, False)
    sp = hdiv.HDiv(topo, ref)
    rng = np.random.default_rng(7500 + 10 * dim + k)
    wV, u = (rng.standard_normal(s).astype(np.float32).astype(np.float64) for s in (sp.n_hdiv, (topo.n_elems, dim, ref.nb)))
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x).reshape(-1), dtype=torch.float32, device=g.device)  # noqa: E731
    y = g.apply_convection(dev(wV), dev(u))
    assert _rel(y, C.apply(topo, ref, sp.to_l2(wV), u, k - 1)) < 1e-6


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("dim,n,k", ORDERS)
def test_apply_every_order(dim, n, k, walls):
    g, topo, ref = _setup(dim, n, k, walls)
    rng = np.random.default_rng(7000 + 100 * dim + 10 * k + walls)
    sp = hdiv.HDiv(topo, ref)
    f32 = lambda x: x.astype(np.float32).astype(np.float64)  # noqa: E731
    wV = f32(rng.standard_normal(sp.n_hdiv))
    w = sp.to_l2(wV)
    u = f32(sp.to_l2(rng.standard_normal(sp.n_hdiv)))  # its own wind below: normal-continuous
    fl = rng.integers(-1, k + 1, size=topo.n_facets).astype(np.int8)
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x).reshape(-1), dtype=torch.float32, device=g.device)  # noqa: E731
    exterior = inlet = None
    if walls:
        b = np.where(topo.boundary)[0][::3]
        vals = rng.standard_normal((1, 1, dim)) * np.ones((b.size, ref.wf.size, 1))   # constant per facet: exact modes
        g.set_inlet(b, vals)
        inlet = np.zeros(topo.n_facets, dtype=bool)
        inlet[b] = True
        ext_u = np.zeros((topo.n_facets, ref.wf.size, dim))
        ext_u[b] = vals
    for wind, same in ((w, False), (u, True)):
        if walls:
            exterior = (ext_u, C.facet_trace(topo, ref, wind, "A"))
        gu, gw = dev(u), dev(wV)
        apply = (lambda: g.apply_convection_l2(gu, gu)) if same else (lambda: g.apply_convection(gw, gu))
        g.set_facet_l(None)
        y = apply()
        assert _rel(y, C.apply(topo, ref, wind, u, k - 1, exterior=exterior, inlet=inlet)) < 1e-6
        g.set_facet_l(torch.as_tensor(fl, device=g.device))
        y = apply()
        assert _rel(y, C.apply(topo, ref, wind, u, fl.astype(np.int64), exterior=exterior, inlet=inlet)) < 1e-6


@pytest.mark.parametrize("dim,n,k", ORDERS)
def test_vjp_per_facet_orders(dim, n, k):
    """The VJP kernels with an order per facet; tolerance of the FP32 VJP parity tests, 2e-6."""
    g, topo, ref = _setup(dim, n, k, False)
    sp = hdiv.HDiv(topo, ref)
    rng = np.random.default_rng(7700 + 10 * dim + k)
    shape = (topo.n_elems, dim, ref.nb)
    wV, u, yb = (rng.standard_normal(s).astype(np.float32).astype(np.float64) for s in (sp.n_hdiv, shape, shape))
    fl = rng.integers(-1, k + 1, size=topo.n_facets).astype(np.int8)
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x).reshape(-1), dtype=torch.float32, device=g.device)  # noqa: E731
    g.set_facet_l(torch.as_tensor(fl, device=g.device))
    wbar, ubar = g.vjp_apply(dev(wV), dev(u), dev(yb))
    wb, ub = A.vjp_apply(topo, ref, sp.to_l2(wV), u, yb, fl.astype(np.int64))
    assert _rel(ubar, ub) < 2e-6
    assert _rel(wbar, sp.dual(wb)) < 2e-6


@pytest.mark.parametrize("n,k,walls", [(3, 3, False), (4, 3, True), (5, 3, False), (3, 4, False), (4, 4, True), (5, 4, False)])
def test_tensor_core_volume_rows(n, k, walls):
    """The tensor-core volume kernel with elements along the rows (variant 6): element counts that
    are no multiple of its tile of 40; the FP32 bounds of the operator (1e-6) and of a substep in
    the parity tests (2e-6)."""
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(3, n)
    rep = None if walls else m.rep
    g = Hopu(m.coords, m.elems, rep, k=k, l=k - 1, prec="f32_tc")
    topo, ref = mesh.MeshTopo(m.coords, m.elems, rep), fe.ref_element(3, k)
    sp = hdiv.HDiv(topo, ref)
    rng = np.random.default_rng(7900 + 10 * n + k)
    u = sp.to_l2(rng.standard_normal(sp.n_hdiv)).astype(np.float32).astype(np.float64)
    g.set_volume_variant(6)
    assert g.tuning_volume()["variant"] == 6
    ud = torch.as_tensor(u.reshape(-1), dtype=torch.float32, device=g.device)
    y = g.apply_convection_l2(ud, ud)
    g.sync()
    assert _rel(y, C.apply(topo, ref, u, u, k - 1)) < 1e-6
    v0 = rng.standard_normal(sp.n_hdiv).astype(np.float32).astype(np.float64)
    a = torch.as_tensor(v0, dtype=torch.float32, device=g.device)
    g.rk_substep(a, 1e-3, 1)
    g.sync()
    assert _rel(a, rk.substeps_stage(sp, v0, 1e-3, 1, k - 1)) < 2e-6
    # a wait that gives up is reported, and the context recovers
    g.set_wait_limit(0)
    g.apply_convection_l2(ud, ud)
    with pytest.raises(Exception, match="volume"):
        g.sync()
    g.clear_error()
    g.set_wait_limit(None)
    assert torch.equal(g.apply_convection_l2(ud, ud), y)
    g.sync()


def test_tensor_core_volume_rows_refused():
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(3, 3)
    for k, prec in ((4, "f32"), (4, "tf32"), (2, "f32_tc"), (5, "f32_tc")):
        g = Hopu(m.coords, m.elems, m.rep, k=k, l=k - 1, prec=prec)
        with pytest.raises(Exception):
            g.set_volume_variant(6)
        g.close()
