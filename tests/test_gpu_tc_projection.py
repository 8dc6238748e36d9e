"""The tensor-core projection by exact digits (k_v2l_tcr) at every order it covers.

Meshes whose element counts are no multiple of its tile of 128, one with several tiles per CTA.
Bound, entry by entry: one rounding of Y, one of the FP32 geometry and d products and sums of the
Piola map, 8 * 2^-24 sum_b |P_ab Y_b| in all; the digits left out of X (2^-32 of the element's
largest functional each) and of the products, KP 2^-31 |P|_1 max|Dinv| max|X|.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fe, hdiv, mesh

pytestmark = pytest.mark.gpu

CASES = [(2, 5, 1), (2, 8, 2), (2, 9, 3), (2, 13, 4), (3, 3, 1), (3, 4, 2), (3, 3, 3), (3, 5, 3), (3, 3, 4), (3, 5, 4),
         (3, 15, 4), (3, 3, 5), (3, 6, 5)]


@pytest.mark.parametrize("dim,n,k", CASES)
def test_projection_by_digits(dim, n, k):
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(dim, n)
    g = Hopu(m.coords, m.elems, m.rep, k=k, l=k - 1, prec="f32_tc", tile_hint=2)
    assert g.tuning()["v2l"] == "tc"
    topo, ref = mesh.MeshTopo(m.coords, m.elems, m.rep), fe.ref_element(dim, k)
    sp = hdiv.HDiv(topo, ref)
    rng = np.random.default_rng(8100 + 100 * dim + 10 * k + n)
    J = np.asarray(topo.J)
    det = np.linalg.det(J)
    P = np.abs(J / det[:, None, None])
    D = np.linalg.inv(np.asarray(sp.Dinv))
    kp, dmax = D.shape[0] + 16, np.abs(np.asarray(sp.Dinv)).max()
    smooth = sp.interpolate(W.taylor_green) + W.uniform_noise(sp.n_hdiv, 1e-3, 0)
    noise = rng.standard_normal(sp.n_hdiv)
    spread = noise * 10.0 ** rng.uniform(-12, 12, sp.n_hdiv)      # every element has its own scale
    for v in (smooth, noise, 1e-30 * noise, 1e30 * noise, spread, 0.0 * noise):
        v = v.astype(np.float32).astype(np.float64)
        out = g.project("hdiv_to_l2", torch.as_tensor(v, dtype=torch.float32, device=g.device))
        g.sync()
        want = sp.to_l2(v)
        Y = np.einsum("eba,eai->ebi", det[:, None, None] * np.linalg.inv(J), want)
        X = np.abs(Y.reshape(len(J), -1) @ D.T).max(axis=1)
        bound = 8 * 2.0 ** -24 * np.einsum("eab,ebi->eai", P, np.abs(Y))
        bound += kp * 2.0 ** -31 * dmax * X[:, None, None] * P.sum(axis=2)[:, :, None]
        err = np.abs(out.double().cpu().numpy().reshape(want.shape) - want)
        assert (err <= bound).all(), float((err / np.maximum(bound, 1e-300)).max())
