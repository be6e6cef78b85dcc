"""Small batches (one block per bundle) against the throughput kernel, which a
call with a fixed lane split takes: every output, bit for bit."""
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


@pytest.fixture(scope="module")
def ctx(pkg):
    c = pkg.Context(0)
    yield c
    c.close()


def _same(a, b):
    for k in a:
        if a[k] is not None:
            assert torch.equal(a[k].view(torch.uint8), b[k].view(torch.uint8)), k


# one warp per set (slots <= 32) against pooled sets, the slot counts at the
# warp edges, two sets (L >= 23), the smallest and largest sizes; plane widths
# 4, 8, 16, 32 with partly filled bundles; more bundles than multiprocessors
PLANAR = [(2, 1, 9), (3, 3, 3), (5, 4, 200), (8, 4, 7), (9, 2, 11), (11, 5, 3), (12, 16, 5), (15, 1, 30), (16, 4, 3),
          (22, 4, 3), (23, 4, 3), (25, 3, 150), (31, 12, 2), (9, 4, 700)]


@pytest.mark.parametrize("L,R,n", PLANAR)
@pytest.mark.parametrize("noise", [0, 1])
def test_planar_equals_throughput_kernel(pkg, ctx, L, R, n, noise):
    p = 0.06 if noise else 0.13
    syn, _ = ctx.gen_syndromes(50 + L, 3, n, L, p, like=torch.zeros(1, device="cuda"), noise=noise)
    kw = dict(chains_per_class=R, n_sweeps=23, burn_in=9, anneal_stages=3, anneal_beta0=0.3, noise=noise,
              beta_scale=0.85 if noise else 1.0)
    a = ctx.decode_ex(syn, L, p, pkg.Opts(**kw), seed=77, id0=3)
    b = ctx.decode_ex(syn, L, p, pkg.Opts(**kw, lanes_per_bundle=32), seed=77, id0=3)
    _same(a, b)
    # resumed from the chains' states and sums at sweep 10
    cut = dict(kw, n_sweeps=10)
    c = ctx.decode_ex(syn, L, p, pkg.Opts(**cut), seed=77, id0=3)
    d = ctx.decode_ex(syn, L, p, pkg.Opts(**kw), seed=77, id0=3, sweep_begin=10, init_frames=c["chain_frames"],
                      init_chain_sum=c["chain_sum"])
    _same(d, b)


@pytest.mark.parametrize("L,R,n", [(2, 1, 5), (4, 4, 3), (8, 1, 33), (16, 2, 3), (30, 4, 2)])
@pytest.mark.parametrize("noise", [0, 1])
def test_toric_equals_throughput_kernel(pkg, ctx, L, R, n, noise):
    p = 0.07
    syn, _ = ctx.gen_syndromes_toric(60 + L, 0, n, L, p, like=torch.zeros(1, device="cuda"))
    kw = dict(n_classes=16, chains_per_class=R, n_sweeps=12, burn_in=4, noise=noise)
    _same(ctx.decode_ex(syn, L, p, pkg.Opts(**kw), seed=5), ctx.decode_ex(syn, L, p, pkg.Opts(**kw, lanes_per_bundle=32), seed=5))


# beta* = 0 (all accepted), low and high temperatures (other digit-plane
# modes), infinity (no uphill step), one sweep, a long run (the counters are
# flushed several times)
@pytest.mark.parametrize("scale,p,sweeps", [(0.0, 0.1, 5), (0.05, 0.1, 9), (0.5, 0.15, 9), (1.0, 0.001, 9), (3.0, 0.1, 9),
                                            (float("inf"), 0.1, 9), (1.0, 0.75, 5), (1.0, 0.15, 1), (1.0, 0.15, 2600)])
def test_temperatures_equal_throughput_kernel(pkg, ctx, scale, p, sweeps):
    L, n = 6, 5
    syn, _ = ctx.gen_syndromes(70, 0, n, L, min(p, 0.3), like=torch.zeros(1, device="cuda"))
    for R in (1, 4, 8):
        kw = dict(chains_per_class=R, n_sweeps=sweeps, burn_in=0, beta_scale=scale)
        _same(ctx.decode_ex(syn, L, p, pkg.Opts(**kw), seed=9),
              ctx.decode_ex(syn, L, p, pkg.Opts(**kw, lanes_per_bundle=32), seed=9))
