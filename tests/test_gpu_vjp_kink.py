"""The cotangent of the wind where w.n is zero to rounding (FP32).

wbar holds sign(w.n) at the facet points.  At a point whose |w.n| is below its own rounding error
the sign is that of the error, so it depends on the order of the sums; the kernels fix one order:
traces by ascending basis index, the normal component by ascending component, then the modes in
order, each step one fused multiply-add.  Here every facet's constant moment is shifted so that w.n
vanishes to rounding at one of its points, and wbar has to be the one with the signs that this order
gives, worked out on the host from the same FP32 wind.

wbar depends on w through these signs alone, so the reference is the oracle's FP64 wbar for winds
moved off the zeros to the given side; a sum that is exactly zero (sign 0) takes the mean of the two
sides.  Facets whose sign hangs on the table's 1e-15 of quadrature rounding (a product half-way
between two FP32 values) keep their wind.  Tolerance: the FP32 bound of the other VJP tests.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import adjoint as A
from oracle import fe, hdiv, mesh

pytestmark = pytest.mark.gpu


def _fma(a, b, c):
    """a b + c in FP32 with one rounding: the product is exact in FP64, the sum is rounded to odd
    there (its last bit set when anything was cut off), so that the step to FP32 is the only rounding."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    cut = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    return np.where((cut != 0) & even, np.nextafter(s, np.where(cut > 0, np.inf, -np.inf)), s).astype(np.float32)


def _wn_fp32(topo, ref, wL, noise):
    """w.n at the facet points in the kernels' order; wL: the FP32 wind [E, d, nb]; noise: what the
    entries of the trace table hold that vanish."""
    d, nf = ref.dim, ref.psi.shape[1]
    trm = np.stack([np.einsum("q,qm,qi->mi", ref.wf, ref.psi, ref.phi_f[f]) for f in range(d + 1)])
    trm = np.where(np.abs(trm) < 1e-12, noise, trm).astype(np.float32)
    side = []
    for ef in (topo.fa, topo.fb):
        t, c = trm[ef[:, 1]], wL[ef[:, 0]]                    # [F, nf, nb], [F, d, nb]
        s = np.zeros((topo.n_facets, nf, d), dtype=np.float32)
        for i in range(ref.nb):
            s = _fma(np.broadcast_to(t[:, :, None, i], s.shape), np.broadcast_to(c[:, None, :, i], s.shape), s)
        side.append(s)
    v = np.float32(0.5) * (side[0] + side[1])
    n = topo.nF.astype(np.float32)
    wn = np.zeros((topo.n_facets, nf), dtype=np.float32)
    for a in range(d):
        wn = _fma(v[:, :, a], np.broadcast_to(n[:, a:a + 1], wn.shape), wn)
    psi = ref.psi.astype(np.float32)
    out = np.zeros((topo.n_facets, psi.shape[0]), dtype=np.float32)
    for m in range(nf):
        out = _fma(np.broadcast_to(psi[:, m], out.shape), np.broadcast_to(wn[:, m:m + 1], out.shape), out)
    return out


@pytest.mark.parametrize("dim,n,k", [(2, 4, 2), (2, 64, 2), (2, 64, 4), (3, 3, 3), (3, 8, 1), (3, 8, 2), (3, 8, 3),
                                     (3, 8, 4), (3, 3, 5), (3, 6, 5)])
def test_wind_cotangent_sign_at_the_kink(dim, n, k):
    from paper_2408_06698_gb300 import Hopu
    m = W.periodic_box_mesh(dim, n)
    g = Hopu(m.coords, m.elems, m.rep, k=k, l=k - 1, prec="f32")
    topo, ref = mesh.MeshTopo(m.coords, m.elems, m.rep), fe.ref_element(dim, k)
    sp = hdiv.HDiv(topo, ref)
    nf, F = ref.psi.shape[1], topo.n_facets
    rng = np.random.default_rng(9100 + 10 * dim + k)
    f32 = lambda x: x.astype(np.float32).astype(np.float64)  # noqa: E731
    wV = f32(rng.standard_normal(sp.n_hdiv))
    u, yb = (f32(rng.standard_normal((topo.n_elems, dim, ref.nb))) for _ in range(2))

    def wn_of(v):
        wL = sp.to_l2(v)
        return A._facet_fields(topo, ref, wL, wL, wL, -1)[1]

    # w.n at point q of facet F moves by unit[F] with the facet's constant moment
    first = np.arange(F) * nf
    one = np.zeros(sp.n_hdiv)
    one[first] = 1.0
    unit = wn_of(one)[:, 0]
    q = rng.integers(0, ref.wf.size, size=F)
    at = np.arange(F), q
    scale = np.abs(wn_of(wV)).mean()
    moved = wV.copy()
    moved[first] -= wn_of(wV)[at] / unit
    moved = f32(moved)
    rest = np.abs(wn_of(moved))
    rest[at] = np.inf
    chosen = rest.min(axis=1) > 1e-3 * scale           # the facet's other points keep their sign
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x).reshape(-1), dtype=torch.float32, device=g.device)  # noqa: E731
    noise = [1e-15 * rng.standard_normal((dim + 1, nf, ref.nb)) for _ in range(10)]
    noise += [-r for r in noise]                       # either way round a half-way product
    while True:                                        # a facet given back moves its neighbours' roundings
        x = wV.copy()
        x[first[chosen]] = moved[first[chosen]]
        wL = g.project("hdiv_to_l2", dev(x)).cpu().numpy().reshape(topo.n_elems, dim, ref.nb)
        signs = [np.sign(_wn_fp32(topo, ref, wL, r)[at]) for r in noise]
        sure = np.all([s == signs[0] for s in signs], axis=0)
        if sure[chosen].all():
            break
        chosen &= sure
    assert chosen.mean() > 0.5
    wV, sign = x, signs[0].astype(np.float64)
    wn = np.abs(wn_of(wV))
    assert wn[at][chosen].max() < 1e-5 * scale
    sides = []
    for zero in (1.0, -1.0):
        x = wV.copy()
        x[first] += np.where(chosen, 1e-4 * scale * np.where(sign == 0, zero, sign) / unit, 0.0)
        sides.append(A.vjp_apply(topo, ref, sp.to_l2(x), u, yb, k - 1)[0])
    want = sp.dual(0.5 * (sides[0] + sides[1]))
    wbar, _ = g.vjp_apply(dev(wV), dev(u), dev(yb))
    got = wbar.double().cpu().numpy()
    err = np.abs(got - want).max() / np.abs(want).max()
    print(f"d={dim} k={k}: {chosen.sum()} points at the kink, {int((sign == 0).sum())} sums of zero, error {err:.2e}")
    assert err < 2e-6
