"""Adam's step against 64 bits, element by element, over the range of the second moment: zero (units that never fired), far below
and far above eps, where the quotient leaves the range of the fast form, and an infinite one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24                       # relative error of one fp32 operation, rounded to nearest


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("eps", [1e-8, 1e-3, 1e-16])
@pytest.mark.parametrize("scale", [1e-16, 1e-10, 1e-3, 1.0, 1e18])
def test_adam_step_against_64_bits(precision, eps, scale):
    import torch
    from paper_2403_11204_b200.binding import Segment
    lr, t0, widths, batch = 1e-3, 5, [157, 200], 64
    seg = Segment(widths, 47, False, precision=precision, optimizer="adam", lr=lr, eps=eps, max_batch=batch, init_seed=2)
    seg.gen_labels(1, "normal")
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand(batch, widths[0], generator=g, device="cuda")
    cls = torch.randint(0, 47, (batch,), generator=g, device="cuda", dtype=torch.int32)
    W, b = [t.clone() for t in seg.params(0)]
    m = torch.randn(W.shape, generator=g, device="cuda") * scale
    v = (torch.rand(W.shape, generator=g, device="cuda") * scale) ** 2
    m[::7], v[::7] = 0, 0
    v[3, 5] = float("inf")
    seg.set_opt_state(0, 0, m, torch.zeros_like(b))
    seg.set_opt_state(0, 1, v, torch.zeros_like(b))
    seg.set_step(t0)
    seg.train_step(x.to(torch.bfloat16) if precision == "bf16" else x, cls)
    seg.poll()
    W0, m0, v0, gw, P, M, V = [t.double().cpu().numpy() for t in
                               (W, m, v, seg.grads(0)[0], seg.params(0)[0], seg.opt_state(0, 0)[0], seg.opt_state(0, 1)[0])]
    b1, b2, l, e = [float(np.float32(c)) for c in (0.9, 0.999, lr, eps)]
    m1, v1 = b1 * m0 + (1 - b1) * gw, b2 * v0 + (1 - b2) * gw * gw
    d = np.sqrt(v1 / (1 - b2 ** (t0 + 1))) + e
    k = l / (1 - b1 ** (t0 + 1)) / d
    # the new parameter's rounding; some twelve rounded operations on the way to the step; the terms of m, which may cancel.  Below
    # 1e-30 (1e-38) products (sums) may have lost bits to the end of fp32's range.
    bound = U * np.maximum(np.abs(W0), np.abs(P)) + 12 * U * np.abs(k * m1) + 4 * U * k * (b1 * np.abs(m0) + (1 - b1) * np.abs(gw)) + 1e-30
    assert np.all(np.abs(P - (W0 - k * m1)) <= bound)
    assert P[3, 5] == W0[3, 5] and np.isinf(V[3, 5])
    np.testing.assert_allclose(M, m1, rtol=0, atol=4 * U * (np.abs(m0) + np.abs(gw)).max())
    seg.close()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_adam_step_outside_the_range_of_its_fast_form(precision):
    """A second moment below zero, however small, has no root; a denominator near the end of fp32's range still divides."""
    import torch
    from paper_2403_11204_b200.binding import Segment
    widths, batch = [157, 200], 64
    x = torch.rand(batch, widths[0], device="cuda")
    cls = torch.zeros(batch, device="cuda", dtype=torch.int32)
    for eps in (1e-8, 1e-3, 3e38):
        seg = Segment(widths, 47, False, precision=precision, optimizer="adam", lr=1.0, eps=eps, max_batch=batch, init_seed=2)
        seg.gen_labels(1, "normal")
        W, b = [t.clone() for t in seg.params(0)]
        m, v = torch.full_like(W, 2e38 if eps > 1 else 0.5), torch.zeros_like(W)
        v[5, :6] = -torch.tensor([1e-41, 2e-38, 1e-36, 1e-33, 1e-20, 1.0], device="cuda")
        b[:] = 1.0
        b[5] = -1.0                                            # never fires: no gradient is added to that row's moments
        seg.set_params(0, torch.zeros_like(W), b)
        seg.set_opt_state(0, 0, m, torch.zeros_like(b))
        seg.set_opt_state(0, 1, v, torch.zeros_like(b))
        seg.set_step(1 << 20)                                  # bias corrections of one
        seg.train_step(x.to(torch.bfloat16) if precision == "bf16" else x, cls)
        seg.poll()
        g, P = seg.grads(0)[0], seg.params(0)[0]
        assert torch.all(g[5] == 0) and torch.any(g != 0)
        assert torch.all(torch.isnan(P) == (v < 0))
        if eps > 1:
            want = -(0.9 * m + 0.1 * g).double() / eps         # -0.6: the root of v is nothing beside eps
            assert torch.all((P.double() - want)[v >= 0].abs() <= 1e-6)
        seg.close()
