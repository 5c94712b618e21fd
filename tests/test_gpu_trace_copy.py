"""Copies of a trace's arrays (gbt_trace_copy): one launch for all of them, 16-byte words where
both ends are aligned and 4-byte words elsewhere.  Bytes: no tolerance."""
import numpy as np
import pytest

from paper_2501_13382_gb300 import inputs as I

pytestmark = pytest.mark.gpu
NAMES = ("ray_off", "o", "t", "L", "s0", "ray", "depth", "bmat", "hit")


@pytest.mark.parametrize("rays", [1, 3, 257, 5000, 70001])
@pytest.mark.parametrize("shift", [0, 1])
def test_copies_are_the_traces_arrays(rays, shift):
    import torch
    from oracle import oracle as O
    from paper_2501_13382_gb300 import gbt as G
    sc0, _ = I.city_scene(I.SEED_BASE + 3)
    src = I.Source(np.array([0.3, -0.2, 3.0]), rays, 3, 600.0)
    tr = G.Trace(G.Scene(sc0), src)
    seg = tr.segments()
    ot = O.trace(sc0, src)
    assert seg["n_segments"] == ot.n_seg
    assert np.array_equal(seg["ray_off"].cpu().numpy(), ot.ray_off)
    # the same through buffers that start `shift` elements into others, one left out
    bufs = {k: torch.full((seg[k].numel() + shift + 1,), -7, dtype=seg[k].dtype, device="cuda")
            for k in NAMES}
    ptr = [bufs[k].data_ptr() + shift * bufs[k].element_size() for k in NAMES]
    ptr[6] = None
    G.gbt_trace_copy(tr.handle, G.gbt_trace_arrays(*ptr), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for k in NAMES:
        b = bufs[k]
        if k == "depth":
            assert bool((b == -7).all())
            continue
        assert torch.equal(b[shift:-1], seg[k].reshape(-1))
        assert bool((b[:shift] == -7).all()) and bool((b[-1:] == -7).all())
