"""Shared-memory limits across calls: a plan of small codes between two decodes
of large ones, on the kernels that read their digit modes from parameters
(partly filled 32-chain bundles)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_2669_gb300 import build as b
    b.build()
    import paper_1302_2669_gb300 as P
    return P


@pytest.mark.parametrize("noise", [0, 1])
def test_plan_of_small_codes_leaves_large_decodes(pkg, noise):
    ctx = pkg.Context(0)
    like = torch.zeros(1, device="cuda")
    opts = pkg.Opts(chains_per_class=9, n_sweeps=4, burn_in=1, lanes_per_bundle=32, noise=noise)
    big, _ = ctx.gen_syndromes(7, 0, 40, 25, 0.1, like=like, noise=noise)
    before = ctx.decode(big, 25, 0.1, opts, seed=3)
    n = 30
    small, _ = ctx.gen_syndromes(8, 0, n, 13, 0.1, like=like, noise=noise)
    cls = torch.empty(n, dtype=torch.int32, device="cuda")
    plan = pkg.RaggedPlan(ctx, np.full(n, 13, np.int32), 0.1, small.reshape(-1), cls, opts=opts, seed=3)
    plan.launch()
    after = ctx.decode(big, 25, 0.1, opts, seed=3)
    torch.cuda.synchronize()
    for a, b in zip(before, after):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert torch.equal(cls, ctx.decode(small, 13, 0.1, opts, seed=3)[0])
    plan.close()
    ctx.close()
