"""Autotuning of parallel banded plans: the plan's own strategy is a candidate with a text of its own, can be asked for
again, and is what every candidate has to beat; a choice cached under the meaning of another version is not applied."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


def uneven(torch):
    """Instances with 3, 40 and 400 rows per column, by explicit row starts: the default differs between them."""
    g = np.random.default_rng(8)
    cols, per = [900, 300, 64], [3, 40, 400]
    start = np.concatenate([np.repeat(np.arange(c), q) for c, q in zip(cols, per)])
    rows = [c * q for c, q in zip(cols, per)]
    left = np.concatenate([np.full(c * q, c) for c, q in zip(cols, per)]) - start
    J = g.standard_normal((sum(rows), 8)).astype(np.float32)
    J[np.arange(8)[None, :] >= left[:, None]] = 0.0
    b = g.standard_normal(sum(rows)).astype(np.float32)
    plan = dict(instance_cols=cols, window=8, solver=2, row_start=start, instance_rows=rows)
    return plan, torch.from_numpy(J.reshape(-1)).cuda(), torch.from_numpy(b).cuda(), sum(cols)


def solution(torch, ctx, J, b, N):
    p = torch.empty(N, device="cuda")
    ctx.factor_solve(J, b, p, lam=1e-3, refine_steps=0)
    ctx.sync_status()
    return p


def test_default_can_be_restored():
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, QRKitError
    plan, J, b, N = uneven(torch)
    ctx = Context(0, precision="fp32")
    ctx.plan_banded(**plan)
    want = solution(torch, ctx, J, b, N)
    ctx.apply_tuning("compress 0 4")
    other = solution(torch, ctx, J, b, N)
    assert not torch.equal(other, want)
    ctx.apply_tuning("compress auto")
    assert torch.equal(solution(torch, ctx, J, b, N), want)
    for bad in ("compress", "compress 0", "compress 0 0", "compress 1 0", "compress 0 65", "compress none"):
        with pytest.raises(QRKitError):
            ctx.apply_tuning(bad)
    assert torch.equal(solution(torch, ctx, J, b, N), want)   # a refused text changes nothing
    ctx.close()


def test_cache_versions(tmp_path):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    plan, J, b, N = uneven(torch)
    p = torch.empty(N, device="cuda")
    texts = ["compress auto", "compress 1 1"] + [f"compress 0 {n}" for n in (2, 4, 8, 16, 32, 64)]

    def tune(cache):
        ctx = Context(0, precision="fp32_refined")
        ctx.plan_banded(**plan)
        choice = ctx.autotune(J, b, p, refine_steps=1, cache_path=cache)
        q = solution(torch, ctx, J, b, N)
        ctx.close()
        return choice, q

    cache = str(tmp_path / "tune.txt")
    choice, q = tune(cache)
    key, text = open(cache).read().strip().split("\t")
    assert choice == text and choice in texts and key.startswith("v3:")
    assert tune(cache)[0] == choice and len(open(cache).read().splitlines()) == 1
    old = str(tmp_path / "old.txt")
    open(old, "w").write("v2:" + key[3:] + "\tcompress 0 3\n")
    assert tune(old)[0] in texts
    lines = open(old).read().splitlines()
    assert len(lines) == 2 and lines[1].startswith(key)   # timed anew
    forced = str(tmp_path / "auto.txt")
    open(forced, "w").write(key + "\tcompress auto\n")
    assert tune(forced)[0] == "compress auto" and len(open(forced).read().splitlines()) == 1
