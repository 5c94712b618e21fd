"""A receiver without a usable position, or one far off the map, among ordinary ones: its warp
and tile go on as if it were not there, in every kernel that forms a frame, a ball or a box of
its receivers.

Tolerances, relative L2 over the ordinary receivers against the FP64 oracle.  FP32: MUFU sine
and cosine err by 3.6e-7 and the phases by a few 2^-24 turns, 2e-6 in all at these sizes; 1e-5
leaves room for terms that cancel.  FP64: the rounding of the complex64 output, 2^-24, as 1e-7.
A receiver 1e7 m away, taken into its neighbours' frame, would cost them 2^-24 of 5e6 m in n."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_13382_gb300 import inputs as I

pytestmark = pytest.mark.gpu
BAD = [np.nan, np.inf, -np.inf, -3e38]


def _case(window):
    sc = I.city_scene(I.SEED_BASE + 3)[0]
    src = I.Source(np.array([0.3, -0.2, 3.0]), 600, 4, 600.0)
    recv = I.random_receivers(np.random.default_rng(4), 130, (-60.0, -60.0, 1.0), (60.0, 60.0, 9.0))
    freqs, b = [250.0, 1000.0], [40.0, 30.0]
    ref = O.gbs_sum(O.trace(sc, src), recv, freqs, b, sc.c, sc.gamma, window=window)
    return sc, src, recv, freqs, b, ref


def _sums(G, tr, r, freqs, b, gam, window, order):
    kw = dict(order=order, window=window)
    return {"plain": (G.gbs_sum(tr, r, freqs, b, gam, **kw), 1e-5),
            "lists": (G.gbs_sum(tr, r, freqs, b, gam, tile_cull=True, **kw), 1e-5),
            "differentiable": (G.gbs_sum_differentiable(tr, r, freqs, b, gam, **kw), 1e-5),
            "differentiable, lists": (G.gbs_sum_differentiable(tr, r, freqs, b, gam, tile_cull=True, **kw), 1e-5),
            "FP64": (G.gbs_sum(tr, r, freqs, b, gam, precision=G.PRECISION_F64, **kw), 1e-7)}


def _worst(got, ref, keep):
    e = got.cpu().numpy()[:, keep].astype(np.complex128) - ref[:, keep]
    return np.linalg.norm(e) / np.linalg.norm(ref[:, keep])


@pytest.mark.parametrize("window", [I.WINDOW_SEGMENT, I.WINDOW_LINE])
@pytest.mark.parametrize("at", [0, 40, 129])
def test_receivers_without_a_position(at, window):
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc, src, recv, freqs, b, ref = _case(window)
    tr = G.Trace(G.Scene(sc), src)
    gam = torch.as_tensor(sc.gamma, device="cuda")
    keep = np.arange(len(recv)) != at
    for axis, bad in enumerate(BAD):
        x = recv.copy()
        x[at, axis % 3] = bad
        r = torch.as_tensor(x, device="cuda")
        for order in (None, G.recv_order(r)):
            for name, (p, tol) in _sums(G, tr, r, freqs, b, gam, window, order).items():
                assert _worst(p, ref, keep) <= tol, (name, bad)
                assert not p[:, at].abs().any(), (name, bad)


def test_gradients_without_a_position():
    """The gradients are those of the sum without the receiver; FP32 sums in any order, 1e-5."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc, src, recv, freqs, b, _ = _case(I.WINDOW_SEGMENT)
    tr = G.Trace(G.Scene(sc), src)
    gam = torch.as_tensor(sc.gamma, device="cuda")
    g = torch.complex(*torch.randn(2, 2, len(recv), generator=torch.Generator().manual_seed(1))).cuda()
    x = recv.copy()
    x[0, 1] = np.nan
    for cull in (False, True):
        kw = dict(window=I.WINDOW_SEGMENT, tile_cull=cull)
        with_it = G.gbs_sum_backward(tr, torch.as_tensor(x, device="cuda"), freqs, b, gam, g, **kw)
        without = G.gbs_sum_backward(tr, torch.as_tensor(x[1:], device="cuda"), freqs, b, gam,
                                     g[:, 1:].contiguous(), **kw)
        for u, v in zip(with_it, without):
            assert float((u.double() - v.double()).norm()) <= 1e-5 * float(v.double().norm())


@pytest.mark.parametrize("at,far", [(0, (1e7, 0.0, 0.0)), (40, (-1e7, 1e7, 2.0)), (129, (3e4, 0.0, -1e4)),
                                    (64, (1e12, 1e12, 0.0))])
def test_one_receiver_far_away(at, far):
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc, src, recv, freqs, b, ref = _case(I.WINDOW_SEGMENT)
    tr = G.Trace(G.Scene(sc), src)
    gam = torch.as_tensor(sc.gamma, device="cuda")
    keep = np.arange(len(recv)) != at
    x = recv.copy()
    x[at] = far
    r = torch.as_tensor(x, device="cuda")
    for cull in (False, True):
        p = G.gbs_sum(tr, r, freqs, b, gam, window=I.WINDOW_SEGMENT, tile_cull=cull)
        assert _worst(p, ref, keep) <= 1e-5, (cull, far)
