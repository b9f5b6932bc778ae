"""LM steps of curve fits of any size: in units 1e-15 or 1e15 times as large, the same iterations (the points' tangents are
of the curve's size, and the damping is relative to the columns of J)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


def run(torch, scale, t, ctrl, data):
    from paper_1802_03773_gb300 import Context
    ctx = Context(0, precision="fp32_refined")
    ctx.lm_plan([t.size], [ctrl.shape[0]], torch.from_numpy(data * scale).cuda())
    x = torch.from_numpy(np.concatenate([t, (ctrl * scale).reshape(-1)])).cuda()
    st = ctx.lm_states(1e-2)
    for _ in range(3):
        ctx.lm_step(x, st, refine_steps=2)
    x = x.cpu().numpy()
    ctx.close()
    return x[:t.size], x[t.size:] / scale, st[0].lambda_


# a power of two scales every operation exactly: the parameters and the damping agree to rounding in double
@pytest.mark.parametrize("power", [-50, 50])
def test_scaled_fit(power):
    torch = cuda_or_skip()
    g = np.random.default_rng(9)
    th = 2 * np.pi * np.arange(12) / 12
    ctrl = np.stack([np.cos(th), np.sin(th)], 1) * (1 + 0.1 * g.standard_normal((12, 1)))
    t = g.random(300) * 9
    data = 0.2 * g.standard_normal((300, 2)) + ctrl[np.minimum(t.astype(int), 8) + 1]
    want, got = run(torch, 1.0, t, ctrl, data), run(torch, 2.0 ** power, t, ctrl, data)
    for a, b in zip(got, want):
        np.testing.assert_allclose(a, b, rtol=1e-9, atol=1e-9 * np.abs(b).max())
