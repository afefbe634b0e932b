"""fit_chi2_sum asks m3e_fit_grad for a gradient exactly where autograd will want one (a stand-in
for the context records the request; no GPU)."""
import pytest

torch = pytest.importorskip("torch")


class _Context:
    def fit_grad(self, hits, off, cand, params, grad=True, stream=None):
        self.asked = grad
        return params.square().sum().reshape(1), 2 * params if grad else None


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("kind", ["parameter", "intermediate", "constant"])
@pytest.mark.parametrize("mode", ["grad", "no_grad", "inference"])
def test_gradient_only_where_it_is_wanted(mode, kind, dtype):
    from paper_2206_11535_gb300 import m3e
    leaf = torch.arange(1.0, 26.0, dtype=dtype)
    if kind != "constant":
        leaf.requires_grad_()
    p = leaf * 1.0 if kind == "intermediate" else leaf
    ctx = _Context()
    with {"grad": torch.enable_grad, "no_grad": torch.no_grad, "inference": torch.inference_mode}[mode]():
        s = m3e.fit_chi2_sum(p, ctx, None, None, None)
    want = mode == "grad" and kind != "constant"
    assert ctx.asked is want and s.requires_grad is want
    assert s.dtype == dtype and s.shape == () and float(s.detach()) == 5525.0
    if want:
        (3.0 * s).backward()
        assert torch.equal(leaf.grad, 6.0 * leaf.detach()) and leaf.grad.dtype == dtype
