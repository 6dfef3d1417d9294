"""The read-out at batch sizes and widths where the number of warps per sample changes.  Against the same formulas in double."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 7, 299, 600, 1200, 2400, 5003])
@pytest.mark.parametrize("F,k,H", [(5, 16, 0), (100, 64, 0), (20, 8, 24), (7, 12, 136), (39, 32, 400)])
def test_logits_and_gradients(B, F, k, H):
    from paper_1909_04823_b200 import binding as D
    g = torch.Generator(device="cuda").manual_seed(B + F + H)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ops = D.OP_LR | D.OP_FM | D.OP_POOL | (D.OP_DENSE1 if H else 0)
    t = D.Table(2, F, k, hidden=H, max_rows=100, max_nnz=64, max_batch=B)
    try:
        hc = dict(b0=-0.5, c_lr=0.75, c_fm=0.25, u=rn(H) / 8 if H else None, b1=rn(H) if H else None, q=None if H else rn(F * k) / 16, d=rn(13))
        out, pooled, Z, x = rn(B, k + 4), rn(B, F * k), rn(B, H) if H else None, rn(B, 13)
        y = (torch.rand(B, generator=g, device="cuda") < 0.3).float()
        logit, loss, gL, gF = (torch.full((B,), 9.0, device="cuda") for _ in range(4))
        gE = torch.full((B, F * k), 9.0, device="cuda") if not H else None
        gZ = torch.full((B, H), 9.0, device="cuda") if H else None
        t.head(ops, B, hc, out, pooled, Z, x, y, logit, loss, gL, gF, gE, gZ)
        z = -0.5 + 0.75 * out[:, k].double() + 0.25 * out[:, k + 1].double() + x.double() @ hc["d"].double()
        if H:
            a = (Z + hc["b1"]).double()                    # (rounded to float32 as the kernel does)
            z = z + a.clamp(min=0) @ hc["u"].double()
        else:
            z = z + pooled.double() @ hc["q"].double()
        p = torch.sigmoid(z)
        ref = (p - y.double()) / B
        close = lambda got, want: bool(((got.double() - want).abs() <= 2e-7 * want.abs() + 1e-12 * want.abs().max() + 1e-30).all())
        assert close(logit, z)
        assert close(loss, torch.nn.functional.binary_cross_entropy_with_logits(z, y.double(), reduction="none"))
        assert close(gL, 0.75 * ref) and close(gF, 0.25 * ref)
        if H:
            assert close(gZ, ref[:, None] * hc["u"].double() * (a > 0))
        else:
            assert close(gE, ref[:, None] * hc["q"].double())
    finally:
        t.close()
