"""The forward pair kernel at the sizes where it can go wrong: edges of warp tiles (64
receivers) and CTA tiles (960), ragged segment batches, every band-slot instantiation, one
and several beam parameters, compact warps (the FP32 projection) and scattered ones (the
split projection), with a segment list and without; and the differentiable sum beside it.

Tolerance: a term's phase moves by at most 3 x 2^-24 x 90 turns = 1.0e-4 rad (the FP32
projection of the differentiable sum at its limit) and its amplitude by a few 2^-22 (MUFU),
independently from term to term, so 1e-4 bounds the relative L2 error also where terms cancel mildly."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_13382_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-4


def _receivers(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "compact":           # a lattice of 2 m near the source's street
        k = int(np.ceil(np.sqrt(n)))
        g = 2.0 * (np.arange(k) - k / 2)
        xx, yy = np.meshgrid(g, g)
        return np.stack([xx.ravel(), yy.ravel(), np.full(k * k, 1.5)], 1)[:n].astype(np.float32)
    return I.random_receivers(rng, n, (-200.0, -200.0, 1.0), (200.0, 200.0, 20.0))


@pytest.mark.parametrize("kind,n,rays,nf,uniform,window,cull", [
    ("compact", 1, 257, 1, True, I.WINDOW_SEGMENT, False),
    ("compact", 63, 300, 2, True, I.WINDOW_SEGMENT, True),
    ("compact", 65, 301, 3, False, I.WINDOW_LINE, False),
    ("compact", 959, 500, 4, True, I.WINDOW_SEGMENT, False),
    ("compact", 961, 333, 6, False, I.WINDOW_SEGMENT, True),
    ("scatter", 64, 1023, 1, True, I.WINDOW_SEGMENT, False),
    ("scatter", 200, 700, 2, False, I.WINDOW_SEGMENT, False),
    ("scatter", 961, 512, 5, True, I.WINDOW_LINE, True),
    ("scatter", 1921, 400, 8, True, I.WINDOW_SEGMENT, False),
    ("scatter", 130, 900, 7, False, I.WINDOW_SEGMENT, True),
])
def test_pair_kernel_edges(kind, n, rays, nf, uniform, window, cull):
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 4, 600.0)
    recv = _receivers(kind, n, rays)
    freqs = list(125.0 * 2.0 ** (np.arange(nf) * (5.0 / max(nf - 1, 1))))[::-1]
    b = [40.0] * nf if uniform else [20.0 + 9.0 * f for f in range(nf)]
    ot = O.trace(sc0, src)
    po = O.gbs_sum(ot, recv, freqs, b, sc0.c, sc0.gamma, window=window)
    sc = G.Scene(sc0)
    tr = G.Trace(sc, src)
    r = torch.as_tensor(recv, device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    args = (tr, r, freqs, b, gam)
    for order in (None, G.recv_order(r)):
        p = G.gbs_sum(*args, order=order, window=window, tile_cull=cull)
        q = G.gbs_sum_differentiable(*args, order=order, window=window, tile_cull=cull)
        torch.cuda.synchronize()
        G.gbt_sync()
        for got in (p, q):
            e = got.cpu().numpy().astype(np.complex128) - po
            assert np.linalg.norm(e) <= TOL * np.linalg.norm(po)


@pytest.mark.parametrize("n,rays,nf,window,cutoff", [
    (1, 257, 1, I.WINDOW_SEGMENT, 16.0),
    (31, 300, 2, I.WINDOW_LINE, 16.0),
    (33, 700, 3, I.WINDOW_SEGMENT, 1e4),
    (65, 1023, 9, I.WINDOW_SEGMENT, 2.0),
    (400, 513, 16, I.WINDOW_LINE, 16.0),
])
def test_f64_kernel_edges(n, rays, nf, window, cutoff):
    """The FP64 sum at the edges of its 32-receiver tiles and candidate windows, with few and
    many bands and with cutoffs that keep few pairs or nearly all.  Tolerance: the complex64
    output rounds each component by at most 2^-24 of it (6e-8 of the L2 norm); FP64 phases of
    up to 1e5 rad add 1e-11."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 4, 600.0)
    recv = _receivers("scatter" if n % 2 else "compact", n, rays)
    freqs = list(125.0 * 2.0 ** (np.arange(nf) * (5.0 / max(nf - 1, 1))))[::-1]
    b = [20.0 + 9.0 * f for f in range(nf)]
    po = O.gbs_sum(O.trace(sc0, src), recv, freqs, b, sc0.c, sc0.gamma, window=window, cutoff=cutoff)
    sc = G.Scene(sc0)
    tr = G.Trace(sc, src)
    r = torch.as_tensor(recv, device="cuda")
    p = G.gbs_sum(tr, r, freqs, b, torch.as_tensor(sc0.gamma, device="cuda"), order=G.recv_order(r),
                  window=window, cutoff=cutoff, precision=G.PRECISION_F64)
    torch.cuda.synchronize()
    e = p.cpu().numpy().astype(np.complex128) - po
    assert np.linalg.norm(e) <= 1e-7 * np.linalg.norm(po)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1024, 1025, 5000, 16383, 16384, 16385, 40001])
def test_receiver_order_is_the_stable_morton_order(n):
    """Counted ranks up to 16,384 receivers, radix passes beyond; codes and order
    from numpy in the same FP32 steps, ties by index.  Integers: no tolerance."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    rng = np.random.default_rng(n)
    x = rng.uniform(-300, 300, (n, 3)).astype(np.float32)
    x[:, 2] = rng.choice(np.float32([1.5, 4.0]), n)
    x[n // 2:] = x[rng.integers(0, max(n // 2, 1), n - n // 2)] if n > 1 else x[n // 2:]   # ties
    lo, hi = x.min(0), x.max(0)
    span = (hi - lo).astype(np.float32)
    u = np.where(span > 0, (x - lo) / np.where(span > 0, span, np.float32(1)), np.float32(0)).astype(np.float32)
    q = np.clip(u * np.float32(1023), 0, 1023).astype(np.uint32)
    code = np.zeros(n, np.uint64)
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1).astype(np.uint64) << np.uint64(3 * b + a)
    got = G.recv_order(torch.as_tensor(x, device="cuda")).cpu().numpy()
    assert np.array_equal(got, np.argsort(code, kind="stable"))


@pytest.mark.parametrize("n,rays,nf,window", [
    (1, 40, 1, I.WINDOW_SEGMENT),
    (960 * 2 + 7, 1500, 2, I.WINDOW_LINE),
    (960 * 25 + 1, 3000, 9, I.WINDOW_SEGMENT),
    (960 * 40, 200, 3, I.WINDOW_SEGMENT),
])
def test_splits_by_list_length_against_equal_splits(n, rays, nf, window):
    """With the pre-cull a tile's number of splits follows its list (one tile and many, empty
    and short lists, two band groups); the same terms as with equal splits, summed in FP32 in
    groups of at most 2,048 and merged exactly: within 2,048 x 2^-24 = 1.2e-4 of the sum, in
    fact far less since rounding errors add at random."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 4, 600.0)
    freqs = list(125.0 * 2.0 ** (np.arange(nf) * (5.0 / max(nf - 1, 1))))
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(_receivers("scatter", n, rays), device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    order = G.recv_order(r)
    auto, equal = (G.gbs_sum(tr, r, freqs, [30.0] * nf, gam, order=order, window=window,
                             tile_cull=True, seg_split=k) for k in (0, 3))
    torch.cuda.synchronize()
    assert float((auto - equal).norm()) <= 1.2e-4 * float(equal.norm())


@pytest.mark.parametrize("cutoff,height,b", [(2.0, 1000.0, 1.0), (0.5, 1000.0, 1.0), (2.0, 5000.0, 0.3)])
def test_f64_candidates_near_an_image_source_seen_from_afar(cutoff, height, b):
    """Receivers a few metres from the image source, on rays whose reflection lies a kilometre
    away: the prefilter's terms alpha |x' - o'|^2 are then far above s^2 + b^2, and their FP32
    rounding must not drop a pair that the FP64 test keeps.  Tolerance: the rounding of the
    complex64 output, 2^-24, and of FP64 phases, 1e-11 of up to 1e5 rad."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0 = I.Scene(I.C_AIR, True, 0.0, 0, np.zeros((0, 3, 3)), np.zeros(0, np.int32),
                  np.zeros(0, np.int32), np.array([0.9], np.float32))
    src = I.Source(np.array([0.2, -0.3, height]), 4000, 1, 4.0 * height)
    rng = np.random.default_rng(9)
    away = rng.uniform(-1.0, 1.0, (96, 3)) * [3.0, 3.0, 2.0] + [0.0, 0.0, 3.0]
    recv = (np.array([0.2, -0.3, -height]) + away).astype(np.float32)
    freqs, bs = [4000.0], [b]
    po = O.gbs_sum(O.trace(sc0, src), recv, freqs, bs, sc0.c, sc0.gamma, window=I.WINDOW_LINE, cutoff=cutoff)
    tr = G.Trace(G.Scene(sc0), src)
    p = G.gbs_sum(tr, torch.as_tensor(recv, device="cuda"), freqs, bs, torch.as_tensor(sc0.gamma, device="cuda"),
                  window=I.WINDOW_LINE, cutoff=cutoff, precision=G.PRECISION_F64)
    torch.cuda.synchronize()
    e = p.cpu().numpy().astype(np.complex128) - po
    assert np.linalg.norm(po) > 0 and np.linalg.norm(e) <= 1e-7 * np.linalg.norm(po)


def test_low_words_of_the_direction_reach_the_phase():
    """One beam at a time (as four equal ones, a group of the plain projection) and two receivers
    4 m either side of a point on it, along x, where K x' is 14 turns and x'.t is exact in FP32: what is left out of t's low word, uniform within
    2^-25 for t_x in [1/2, 1), turns up in the phase as 14 x 2 pi x 2^-25 / sqrt(3) = 1.5e-6 rad
    rms.  With it the phase errs by MUFU's sine and cosine (3.6e-7 at most) and four roundings of
    at most 2^-25 turns, 3.4e-7 rms together if all were at their worst; the bar is 6e-7."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0 = I.Scene(I.C_AIR, False, 0.0, 0, np.zeros((0, 3, 3)), np.zeros(0, np.int32),
                  np.zeros(0, np.int32), np.array([1.0], np.float32))
    sc = G.Scene(sc0)
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    rng = np.random.default_rng(2)
    freqs, b = [3.5 * I.C_AIR], [100.0]
    err = []
    for _ in range(200):
        d = rng.normal(size=3)
        d[0] = abs(d[0]) + np.hypot(d[1], d[2]) * 0.8
        d /= np.linalg.norm(d)
        c = np.round(8.0 * 90.0 * d) / 8.0
        recv = (c + np.array([[4.0, 0.0, 0.0], [-4.0, 0.0, 0.0]])).astype(np.float32)
        src = I.Source(np.zeros(3), 4, 0, 1000.0)
        dirs = np.tile(d, (4, 1))
        po = O.gbs_sum(O.trace(sc0, src, dirs=dirs), recv, freqs, b, sc0.c, sc0.gamma, window=I.WINDOW_LINE)
        tr = G.Trace(sc, src, dirs=torch.as_tensor(dirs, device="cuda"))
        p = G.gbs_sum(tr, torch.as_tensor(recv, device="cuda"), freqs, b, gam, window=I.WINDOW_LINE)
        err.append(np.angle(p.cpu().numpy().astype(np.complex128) / po).ravel())
    rms = np.sqrt(np.mean(np.square(err)))
    assert rms <= 6e-7, rms


@pytest.mark.parametrize("scene,window,nf", [("city", I.WINDOW_SEGMENT, 3), ("city", I.WINDOW_LINE, 1),
                                             ("plane", I.WINDOW_LINE, 6)])
def test_fields_against_a_sum_that_skips_nothing(scene, window, nf):
    """The FP32 field without lists, with lists and with explicit splits, at a sample of the
    receivers, against the oracle, which tests every pair: a segment that a ball test, a list or a
    split drops or takes twice shows here.  1e-6: the worst of MUFU (3.6e-7), the projection and
    the FP32 sums is under it, a beam lost at the cutoff's edge (e^-16 of its peak) not."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    if scene == "city":
        w = I.city(n_rays=32768, n_recv_side=96)
        sc0, src, recv = w.scene, w.sources[0], w.receivers
    else:
        w = I.open_plane_large()
        sc0, src, recv = w.scene, w.sources[0], w.receivers[::3]
    freqs = [500.0 * 2.0 ** (3.0 * f / max(nf - 1, 1)) for f in range(nf)]
    b = [100.0 - 7.0 * f for f in range(nf)]
    some = np.sort(np.random.default_rng(3).permutation(len(recv))[:150])
    po = O.gbs_sum(O.trace(sc0, src), recv[some], freqs, b, sc0.c, sc0.gamma, window=window)
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(np.ascontiguousarray(recv, np.float32), device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    order = G.recv_order(r)
    for kw in (dict(), dict(tile_cull=True), dict(seg_split=7), dict(tile_cull=True, seg_split=7),
               dict(order=None)):
        p = G.gbs_sum(tr, r, freqs, b, gam, window=window, **{"order": order, **kw})
        e = p.cpu().numpy()[:, some].astype(np.complex128) - po
        assert np.linalg.norm(e) <= 1e-6 * np.linalg.norm(po), kw


@pytest.mark.parametrize("nf,n", [(1, 700), (3, 1930)])
def test_differentiable_sum_repeats_and_regroups(nf, n):
    """The differentiable sum repeats to the bit, with lists and without; the two differ by the
    rounding of FP32 sums in other groups of at most 512 terms, at random: 1e-6."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), 3000, 4, 600.0)
    freqs = list(250.0 * 2.0 ** np.arange(nf))
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(_receivers("scatter", n, 5), device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    kw = dict(order=G.recv_order(r), window=I.WINDOW_SEGMENT)
    a, b, c, d = (G.gbs_sum_differentiable(tr, r, freqs, [40.0] * nf, gam, tile_cull=cull, **kw)
                  for cull in (False, False, True, True))
    assert torch.equal(a, b) and torch.equal(c, d)
    assert float((a - c).norm()) <= 1e-6 * float(a.norm())


@pytest.mark.parametrize("kind,n,rays,nf,uniform,window", [
    ("compact", 1, 257, 1, True, I.WINDOW_SEGMENT),
    ("compact", 65, 301, 3, False, I.WINDOW_LINE),
    ("compact", 959, 500, 1, True, I.WINDOW_SEGMENT),
    ("compact", 961, 333, 6, False, I.WINDOW_SEGMENT),
    ("scatter", 64, 1023, 1, True, I.WINDOW_SEGMENT),
    ("scatter", 961, 512, 5, True, I.WINDOW_LINE),
    ("scatter", 1921, 400, 8, True, I.WINDOW_SEGMENT),
    ("scatter", 130, 900, 7, False, I.WINDOW_SEGMENT),
])
def test_forward_field_to_a_few_roundings(kind, n, rays, nf, uniform, window):
    """The forward sum at edges of its tiles and band slots, with lists, splits by list length
    and equal splits, far under the bar of the differentiable sum.  A term's phase errs by MUFU
    (3.6e-7) and some six roundings of 2^-25 turns (1.1e-6 rad), its amplitude by 6e-7 (ex2, rcp):
    2e-6 at worst, which mild cancellation of terms may double; 5e-6.  One band on a compact warp
    adds 3 x 2^-24 x 8 turns at worst, 9e-6 rad, independently from term to term."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 4, 600.0)
    recv = _receivers(kind, n, rays)
    freqs = list(125.0 * 2.0 ** (np.arange(nf) * (5.0 / max(nf - 1, 1))))[::-1]
    b = [40.0] * nf if uniform else [20.0 + 9.0 * f for f in range(nf)]
    po = O.gbs_sum(O.trace(sc0, src), recv, freqs, b, sc0.c, sc0.gamma, window=window)
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(recv, device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    for kw in (dict(), dict(tile_cull=True), dict(tile_cull=True, seg_split=3)):
        p = G.gbs_sum(tr, r, freqs, b, gam, order=G.recv_order(r), window=window, **kw)
        out = torch.ones_like(p)
        G.gbs_sum(tr, r, freqs, b, gam, order=G.recv_order(r), window=window, out=out, accumulate=True, **kw)
        for q, ref in ((p, po), (out, po + 1.0)):
            e = q.cpu().numpy().astype(np.complex128) - ref
            assert np.linalg.norm(e) <= 5e-6 * np.linalg.norm(ref), kw


@pytest.mark.parametrize("n,nf,uniform,window,cutoff,lossy", [
    (1, 1, True, I.WINDOW_SEGMENT, 16.0, False),
    (63, 2, False, I.WINDOW_SEGMENT, 2.0, False),
    (65, 3, True, I.WINDOW_LINE, 16.0, False),
    (130, 6, False, I.WINDOW_SEGMENT, 16.0, False),
    (961, 8, True, I.WINDOW_SEGMENT, 1e4, False),
    (700, 8, False, I.WINDOW_LINE, 16.0, True),
    (2000, 1, True, I.WINDOW_LINE, 0.5, True),
    (1000, 11, True, I.WINDOW_SEGMENT, 16.0, True),
])
def test_receivers_without_an_order(n, nf, uniform, window, cutoff, lossy):
    """Receivers in no order go through candidates of their own where beams are small against
    their warp tile; the same receivers in the order given (the identity) do not.  Both against
    the oracle to 5e-6 (see test_forward_field_to_a_few_roundings; the tiles are 250 m wide, where
    n errs by 2^-24 of that), wide and narrow cutoffs, every band slot."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), 900, 4, 600.0)
    recv = _receivers("scatter", n, 11 + n)
    freqs = list(250.0 * 2.0 ** (np.arange(nf) * (4.0 / max(nf - 1, 1))))
    b = [40.0] * nf if uniform else [20.0 + 9.0 * f for f in range(nf)]
    absorption = [1e-3 * (1 + f) for f in range(nf)] if lossy else None
    ot = O.trace(sc0, src)
    po = O.gbs_sum(ot, recv, freqs, b, sc0.c, sc0.gamma, window=window, cutoff=cutoff, absorption=absorption)
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(recv, device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    for order in (None, torch.arange(n, dtype=torch.int32, device="cuda")):
        p = G.gbs_sum(tr, r, freqs, b, gam, order=order, window=window, cutoff=cutoff, absorption=absorption)
        e = p.cpu().numpy().astype(np.complex128) - po
        assert np.linalg.norm(e) <= 5e-6 * np.linalg.norm(po), order is None


@pytest.mark.parametrize("nf", [7, 8, 9, 10, 15, 16])
@pytest.mark.parametrize("uniform", [True, False])
def test_every_band_of_every_group(nf, uniform):
    """More than eight bands run as groups of at most eight, the last of which may hold one band:
    each band by itself against the oracle, with equal and unequal beam parameters, with lists,
    without an order, and differentiable.  5e-6 as for the forward field, per band."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), 3000, 3, 500.0)
    recv = _receivers("compact", 150, 3)
    freqs = list(125.0 * 2.0 ** (np.arange(nf) * (4.0 / (nf - 1))))
    b = [40.0] * nf if uniform else [100.0 / (1.0 + 0.3 * f) for f in range(nf)]
    po = O.gbs_sum(O.trace(sc0, src), recv, freqs, b, sc0.c, sc0.gamma, window=I.WINDOW_SEGMENT)
    tr = G.Trace(G.Scene(sc0), src)
    r = torch.as_tensor(recv, device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    o = G.recv_order(r)
    for name, p in [("plain", G.gbs_sum(tr, r, freqs, b, gam, order=o, window=I.WINDOW_SEGMENT)),
                    ("lists", G.gbs_sum(tr, r, freqs, b, gam, order=o, window=I.WINDOW_SEGMENT, tile_cull=True)),
                    ("no order", G.gbs_sum(tr, r, freqs, b, gam, window=I.WINDOW_SEGMENT)),
                    ("differentiable", G.gbs_sum_differentiable(tr, r, freqs, b, gam, order=o,
                                                                window=I.WINDOW_SEGMENT))]:
        e = p.cpu().numpy().astype(np.complex128) - po
        rel = np.linalg.norm(e, axis=1) / np.linalg.norm(po, axis=1)
        assert rel.max() <= 5e-6, (name, rel)


@pytest.mark.parametrize("n,nf,window", [(65, 1, I.WINDOW_SEGMENT), (700, 3, I.WINDOW_LINE), (1500, 8, I.WINDOW_SEGMENT)])
def test_differentiable_sum_is_the_same_without_an_order(n, nf, window):
    """Without an order the differentiable sum gives each receiver its own candidates; given the
    identity as an order it does not.  The same terms in the same order: the same bits."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    tr = G.Trace(G.Scene(sc0), I.Source(np.array([0.3, -0.2, 3.0]), 1500, 4, 600.0))
    r = torch.as_tensor(_receivers("scatter", n, 2), device="cuda")
    gam = torch.as_tensor(sc0.gamma, device="cuda")
    freqs = list(500.0 * 2.0 ** (np.arange(nf) / 2.0))
    a, b = (G.gbs_sum_differentiable(tr, r, freqs, [30.0] * nf, gam, order=o, window=window)
            for o in (None, torch.arange(n, dtype=torch.int32, device="cuda")))
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
