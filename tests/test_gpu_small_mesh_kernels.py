"""Separate wind in FP32 on both sides of the mesh sizes at which the kernels change.

On small meshes the facet term and the VJP run a warp per facet or element, on larger ones the register
kernels.  For every order that has such a line: a mesh on each side of it, random data, walls and
per-facet orders for the apply, against the FP64 oracle at the bounds of the other tests (apply 1e-6,
VJP 2e-6 of the largest entry).
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import adjoint as A
from oracle import convection as C
from oracle import fe, hdiv, mesh

pytestmark = pytest.mark.gpu


def _setup(dim, n, k, walls=False):
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(dim, n)
    rep = None if walls else m.rep
    g = Hopu(m.coords, m.elems, rep, k=k, l=k - 1, prec="f32")
    topo = mesh.MeshTopo(m.coords, m.elems, rep)
    sp = hdiv.HDiv(topo, fe.ref_element(dim, k))
    rng = np.random.default_rng(8800 + 100 * dim + 10 * k + n)
    f32 = lambda x: x.astype(np.float32).astype(np.float64)  # noqa: E731
    wV = f32(rng.standard_normal(sp.n_hdiv))
    u, y = (f32(rng.standard_normal((topo.n_elems, dim, sp.ref.nb))) for _ in range(2))
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x).reshape(-1), dtype=torch.float32, device=g.device)  # noqa: E731
    return g, sp, rng, wV, u, y, dev


def _rel(got, ref):
    got = got.double().cpu().numpy().reshape(-1)
    return float(np.abs(got - np.asarray(ref).reshape(-1)).max() / np.abs(ref).max())


# facets: 8 (2D), 12 and 4 (3D) per SM
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("dim,n,k", [(2, 20, 3), (2, 21, 3), (2, 20, 4), (2, 21, 4), (3, 5, 4), (3, 6, 4), (3, 3, 5), (3, 4, 5)])
def test_facet_term(dim, n, k, walls):
    g, sp, rng, wV, u, _, dev = _setup(dim, n, k, walls)
    topo, ref = sp.topo, sp.ref
    fl = rng.integers(-1, k + 1, size=topo.n_facets).astype(np.int8)
    gfl = torch.as_tensor(fl, device=g.device)
    want = C.apply(topo, ref, sp.to_l2(wV), u, fl.astype(np.int64))
    assert _rel(g.apply_convection(dev(wV), dev(u), facet_l=gfl), want) < 1e-6


# elements: 4 (k = 1), 8 (2D k = 2) and 32 per SM; facets: 10 per SM (2D k = 4, 3D k = 2)
@pytest.mark.parametrize("dim,n,k", [(2, 17, 1), (2, 18, 1), (2, 24, 2), (2, 25, 2), (2, 49, 3), (2, 50, 3), (2, 22, 4), (2, 23, 4),
                                     (2, 49, 4), (2, 50, 4), (3, 4, 1), (3, 5, 1), (3, 5, 2), (3, 6, 2), (3, 9, 2), (3, 10, 2)])
def test_vjp(dim, n, k):
    g, sp, _, wV, u, y, dev = _setup(dim, n, k)
    w_ref, u_ref = A.vjp_apply(sp.topo, sp.ref, sp.to_l2(wV), u, y, k - 1)
    w_ref = sp.dual(w_ref)
    wbar, ubar = g.vjp_apply(dev(wV), dev(u), dev(y))
    assert _rel(wbar, w_ref) < 2e-6 and _rel(ubar, u_ref) < 2e-6
    # one cotangent alone: the same kernels
    assert torch.equal(g.vjp_apply(dev(wV), dev(u), dev(y), need_u=False)[0], wbar)
    assert torch.equal(g.vjp_apply(dev(wV), dev(u), dev(y), need_w=False)[1], ubar)
