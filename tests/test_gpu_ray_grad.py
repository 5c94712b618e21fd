"""The parameter gradients of a ray (gamma per bounce, weight per ray, beam parameter per band)
from its segments' gradients: the band counts of each instantiation, a gamma of zero in the
middle of paths, and a weight that is not a number on rays without any gradient.  Bar: 1e-3
relative, the adjoint's (its segments' gradients are FP32 sums in any order)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_13382_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-3


@pytest.mark.parametrize("nf,zero", [(1, False), (2, True), (4, False), (5, True), (8, False)])
def test_ray_gradients(nf, zero):
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0 = I.diff_city().scene
    rng = np.random.default_rng(nf)
    gamma = rng.uniform(0.6, 0.95, sc0.gamma.shape[0]).astype(np.float32)
    if zero:
        gamma[-1] = 0.0
    src = I.Source(I.diff_city().sources[0].pos, 4001, 6, 1000.0)
    recv = I.receiver_grid(13, 120.0, 1.5)
    freqs = 250.0 * (1.0 + np.arange(nf))
    b = np.array([I.beam_b_rule(src.n_rays, f) for f in freqs])
    otr = O.trace(sc0, src)
    po = O.gbs_sum(otr, recv, freqs, b, sc0.c, gamma, window=I.WINDOW_SEGMENT)
    cot = (rng.normal(size=po.shape) + 1j * rng.normal(size=po.shape)) * np.abs(po).mean()
    want = O.gbs_adjoint(otr, recv, freqs, b, sc0.c, gamma, cot, window=I.WINDOW_SEGMENT)
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(recv, device="cuda")
    args = (tr, r, list(freqs), list(b), torch.as_tensor(gamma, device="cuda"),
            torch.as_tensor(cot.astype(np.complex64), device="cuda"))
    got = G.gbs_sum_backward(*args, order=G.recv_order(r), window=I.WINDOW_SEGMENT)
    torch.cuda.synchronize()
    for x, y in zip((got[0], got[1], got[2]), want):
        assert np.linalg.norm(x.cpu().numpy() - y) <= TOL * np.linalg.norm(y)
    # rays that reach no receiver add nothing, whatever their weight
    idle = got[1] == 0
    assert bool(idle.any())
    w = torch.full((src.n_rays,), 4 * np.pi / src.n_rays, dtype=torch.float32, device="cuda")
    for fill in (float("nan"), float("inf")):
        w2 = torch.where(idle, torch.full_like(w, fill), w)
        dg, _, db = G.gbs_sum_backward(*args, ray_weight=w2, order=G.recv_order(r),
                                       window=I.WINDOW_SEGMENT)
        dg0, _, db0 = G.gbs_sum_backward(*args, ray_weight=w, order=G.recv_order(r),
                                         window=I.WINDOW_SEGMENT)
        assert float((dg - dg0).norm()) <= 1e-5 * float(dg0.norm())
        assert float((db - db0).norm()) <= 1e-5 * float(db0.norm())
