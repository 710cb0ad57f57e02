"""The front end's threshold, found by a radix select, where it can go wrong:
ties, one valid pixel, both order statistics under one prefix or not, the first
and last rank, images smaller and larger than a block of 1024 pixels. Pixels,
points and features must equal oracle/frontend.py bit for bit."""
import numpy as np
import pytest

from oracle import frontend

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cvo():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1904_02266_gb300 as m
    return m


def _image(kind, W, H):
    rng = np.random.default_rng(W * 1009 + H)
    depth = rng.uniform(0.6, 4.9, (H, W)).astype(np.float32)
    hsv = rng.random((H, W, 3)).astype(np.float32)
    if kind == "steps":        # few distinct magnitudes: ties at the threshold
        hsv[..., 2] = np.round(hsv[..., 2] * 2) / 2
    elif kind == "flat":       # every magnitude zero
        hsv[..., 2] = 0.25
    elif kind == "fine":       # magnitudes that differ in their last bits
        hsv[..., 2] = np.float32(0.5) + (np.arange(W) % 2 * 1.0 + rng.random((H, W)) * 1e-6)
    elif kind == "sparse":     # mostly without depth
        depth[rng.random((H, W)) < 0.98] = 0.0
    elif kind == "one":
        depth[:] = 9.0
        depth[H // 2, W // 2] = 1.0
    return depth, hsv


@pytest.mark.parametrize("kind", ["noise", "steps", "flat", "fine", "sparse", "one"])
@pytest.mark.parametrize("W,H", [(2, 2), (33, 31), (32, 32), (1025, 3), (200, 150)])
def test_threshold_edges(cvo, kind, W, H):
    torch = pytest.importorskip("torch")
    depth, hsv = _image(kind, W, H)
    if not ((depth >= 0.5) & (depth <= 5.0)).any():
        depth[0, 0] = 1.0
    out = [torch.zeros((W * H, c), dtype=torch.float32, device="cuda") for c in (3, 5)]
    pix = torch.zeros(W * H, dtype=torch.int32, device="cuda")
    with cvo.Context(device=0) as ctx:
        for q, cap in ((0.0, 0), (37.5, 0), (80.0, 7), (99.9, 0), (100.0, 0)):
            fp = cvo.cvo_frontend_params_default(cx=W / 2, cy=H / 2, percentile=q, max_points=cap)
            n = ctx.frontend_select(depth, hsv, fp, out[0], out[1], pix)
            torch.cuda.synchronize()
            xyz, feat, idx = frontend.select(depth, hsv, 525.0, 525.0, W / 2, H / 2, percentile=q,
                                             max_points=cap)
            assert n == idx.size, (q, cap)
            assert np.array_equal(pix[:n].cpu().numpy().astype(np.int64), idx)
            assert np.array_equal(out[0][:n].cpu().numpy(), xyz)
            assert np.array_equal(out[1][:n].cpu().numpy(), feat)
