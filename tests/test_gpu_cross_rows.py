"""The cross layer's rows-in-registers kernels (no per-shard scalars asked for) at the edges of their layouts: one warp per
row, several, rows of a group past the batch's end, the longest row, and the shapes that fall back."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _close(got, ref, tol, what):
    bad = np.abs(got.cpu().numpy().astype(np.float64) - ref) > tol
    assert not bad.any(), (what, int(bad.sum()), float(np.abs(got.cpu().numpy() - ref).max()))


@pytest.mark.parametrize("d", [4, 64, 128, 132, 512, 1020, 1250, 1248, 2048, 2052])
@pytest.mark.parametrize("B", [1, 5, 333, 5000])
def test_rows_in_registers(B, d):
    from paper_1909_04823_b200 import binding
    rng = np.random.default_rng([B, d])
    x0, x, gY = (rng.standard_normal((B, d)).astype(np.float32) for _ in range(3))
    w = (rng.standard_normal(d) / np.sqrt(d)).astype(np.float32)
    b = rng.standard_normal(d).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    y, P, part = binding.cross_forward(dev(x0), dev(x), dev(w), dev(b), min(d, 3))
    assert part is None
    ref = oracle.cross_forward(x0, x, w, b, min(d, 3))
    e = 2e-6 * ref["Sabs"]                             # float32 dot product: a few roundings of the summands' size
    _close(P, ref["P"], 1e-6 + 1e-5 * np.abs(ref["P"]) + e, "P")
    _close(y, ref["y"], 1e-6 + 1e-5 * np.abs(ref["y"]) + np.abs(x0) * e[:, None], "y")
    P32 = ref["P"].astype(np.float32)
    gx0, gx, gw, gb = binding.cross_backward(dev(x0), dev(x), dev(w), dev(P32), dev(gY))
    rb = oracle.cross_backward(x0, x, w, P32, gY)
    t = 2e-6 * np.sum(np.abs(gY.astype(np.float64) * x0), axis=1)
    _close(gx0, rb["gx0"], 1e-6 + 1e-5 * np.abs(rb["gx0"]), "gx0")
    _close(gx, rb["gx"], 1e-6 + 1e-5 * np.abs(rb["gx"]) + np.abs(w)[None] * t[:, None], "gx")
    tx = np.abs(rb["t"])[:, None] * np.abs(x)
    _close(gw, rb["gw"], 1e-6 + 1e-5 * np.abs(rb["gw"]) + 2e-6 * tx.sum(0) + (t[:, None] * np.abs(x)).sum(0), "gw")
    _close(gb, rb["gb"], 1e-6 + 1e-5 * np.abs(rb["gb"]) + 2e-6 * np.abs(gY).sum(0), "gb")
