"""surfmcmc_sweep_time: the time of overlapping launches counts once, every
launch counts."""
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


# n: one block per bundle, many streams on the throughput kernel, one stream
# (7,500 bundles of 32 lanes fill the device twice)
@pytest.mark.parametrize("n", [2, 1000, 15000])
@pytest.mark.parametrize("stages", [0, 2])
def test_ti_time_within_the_call(pkg, n, stages):
    L, p, n_beta = 9, 0.12, 21
    ctx = pkg.Context(0)
    syn, _ = ctx.gen_syndromes(3, 0, n, L, p, like=torch.zeros(1, device="cuda"))
    opts = pkg.Opts(chains_per_class=4, n_sweeps=20, burn_in=5, anneal_stages=stages, anneal_beta0=0.5 if stages else 1.0,
                    lanes_per_bundle=32 if n == 15000 else 0)
    ctx.decode_ti(syn, L, p, opts, n_beta=n_beta, seed=1)
    ctx.set_timing(True)
    ctx.sweep_time()
    a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    ctx.decode_ti(syn, L, p, opts, n_beta=n_beta, seed=1)
    e.record()
    e.synchronize()
    ms, launches = ctx.sweep_time()
    assert launches == (n_beta - 1) * (stages + 1)
    # the sweeps are nearly all of the call, and inside it
    assert 0.3 * a.elapsed_time(e) < ms <= a.elapsed_time(e)
    ctx.set_timing(False)
    ctx.close()
