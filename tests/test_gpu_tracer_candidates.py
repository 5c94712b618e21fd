"""The BVH tracer keeps FP32 bounds during the traversal and tests what is left in FP64
afterwards; the index-order search tests every triangle in FP64 as it goes.  Their traces
must be the same to the bit also where the bounds decide nothing: stacks of coincident
triangles (more than the four candidates a ray keeps), sheets closer together than the FP32
bounds resolve, rays through shared edges and corners, and walls that meet the ground."""
import numpy as np
import pytest

from paper_2501_13382_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _scene(stack, gap, seed):
    rng = np.random.default_rng(seed)
    tri = []
    for q in range(6):                   # quads around the source, each a stack of sheets
        c, s = np.cos(q * np.pi / 3), np.sin(q * np.pi / 3)
        for k in range(stack):
            d = 20.0 + gap * k
            a = np.array([d * c + 15 * s, d * s - 15 * c, 0.0])
            b = np.array([d * c - 15 * s, d * s + 15 * c, 0.0])
            up = np.array([0.0, 0.0, 12.0])
            tri += [(a, b, b + up), (a, b + up, a + up)]
    for _ in range(8):                   # and slivers anywhere
        p = rng.uniform(-15, 15, 3) + [0, 0, 16]
        tri.append((p, p + rng.uniform(-8, 8, 3), p + rng.uniform(-1e-3, 1e-3, 3)))
    tri = np.array(tri)
    n = len(tri)
    return I.Scene(I.C_AIR, True, 0.0, 0, tri, np.ones(n, np.int32), np.arange(n, dtype=np.int32),
                   np.array([1.0, 0.9], np.float32))


@pytest.mark.parametrize("stack,gap", [(1, 0.0), (4, 0.0), (5, 0.0), (9, 0.0), (5, 1e-4), (6, 1e-2),
                                       (3, 0.5)])
def test_bvh_candidates_match_index_order(stack, gap):
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc = _scene(stack, gap, 7 + stack)
    dirs = np.random.default_rng(5).normal(size=(4096, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    # exactly at shared edges and corners of the first wall
    dirs[:8] = np.array([[20, 15, 6], [20, -15, 0], [20, 0, 0], [20, 15, 12], [20, 15, 0],
                         [0, 0, -1], [0, 0, 1], [1, 0, 0]]) - [0, 0, 2] * np.array([[1]] * 5 + [[0]] * 3)
    dirs[:8] /= np.linalg.norm(dirs[:8], axis=1, keepdims=True)
    src = I.Source(np.array([0.0, 0.0, 2.0]), len(dirs), 6, 500.0)
    got = []
    for accel in (G.ACCEL_BVH, G.ACCEL_LINEAR):
        t = G.Trace(G.Scene(sc, accel=accel), src, dirs=torch.as_tensor(dirs, device="cuda"))
        got.append(t.segments())
    G.gbt_sync()
    assert got[0]["n_segments"] == got[1]["n_segments"]
    for k in ("ray_off", "hit", "bmat", "o", "t", "L", "s0"):
        assert torch.equal(got[0][k], got[1][k]), k


@pytest.mark.parametrize("rays", [1, 31, 8191, 8209, 16500, 33001, 66003, 132001])
def test_strips_of_any_length_match_index_order(rays):
    """One ray of a strip up to 32 by the number of rays; the same segments, to the bit."""
    import torch
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 5, 700.0)
    a, b = (G.Trace(G.Scene(sc0, accel=m), src).segments() for m in (G.ACCEL_BVH, G.ACCEL_LINEAR))
    G.gbt_sync()
    assert a["n_segments"] == b["n_segments"]
    for k in ("ray_off", "o", "t", "L", "s0", "ray", "depth", "bmat", "hit"):
        assert torch.equal(a[k], b[k]), k
