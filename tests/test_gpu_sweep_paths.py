"""The paths that full batches take, against the oracle, bit for bit: the
throughput kernel at every lane split, plane width and digit pattern (a call
with fixed lanes never runs one block per bundle), thermodynamic integration
on one and on several streams, and captured plans on either kernel."""
import numpy as np
import pytest

import oracle as O

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


# error rates and beta* scales of the four compiled digit patterns: the first
# eight binary digits of T[1..4] as (none, T1), (T1, T1 and T2), (any, any),
# (T1, any)
TEMPS = {0: [(0.13, 1.0), (0.17, 1.0), (0.13, 0.4), (0.13, 0.5)],
         1: [(0.05, 1.0), (0.08, 1.0), (0.05, 0.4), (0.05, 0.5)]}


# R: planes of 4, 8, 16 and 32 chains, the last also partly filled (9); n
# leaves bundles and warps partly filled
@pytest.mark.parametrize("noise", [0, 1])
@pytest.mark.parametrize("R", [1, 2, 4, 9, 16])
@pytest.mark.parametrize("lanes", [2, 4, 8, 16, 32])
def test_throughput_kernel_equals_oracle(pkg, ctx, lanes, R, noise):
    L, n, sweeps, burn = 7, 5, 9, 3
    for p, scale in TEMPS[noise]:
        syn, _ = O.gen_syndromes(4000 + R, 0, n, L, p, noise)
        opts = pkg.Opts(chains_per_class=R, n_sweeps=sweeps, burn_in=burn, beta_scale=scale, noise=noise,
                        lanes_per_bundle=lanes)
        out = ctx.decode_ex(torch.from_numpy(syn).cuda(), L, p, opts, seed=19, id0=6)
        for i in range(n):
            ref = O.decode_one(L, p, 4, R, sweeps, 19, 6 + i, syn[i], burn_in=burn, beta_scale=scale, noise=noise)
            assert int(out["cls"][i]) == ref["cls"]
            for k in ("class_sum", "log_ratio", "chain_sum", "chain_n"):
                assert (out[k][i].cpu().numpy() == ref[k]).all(), k
            fr = out["chain_frames"][i].cpu().numpy()
            assert (fr[:, 0, :] == O.pack_bits(ref["frames_x"])).all()
            assert (fr[:, 1, :] == O.pack_bits(ref["frames_z"])).all()


# (16 grid points at a time; one after the other: 15,000 syndromes are 1,875
# units of 32 lanes, more than twice what the device holds)
@pytest.mark.parametrize("L,n,n_beta,lanes", [(5, 130, 21, 0), (5, 400, 21, 32), (3, 15000, 5, 32)])
def test_ti_streams_equal_oracle(pkg, ctx, L, n, n_beta, lanes):
    p, R, sweeps, burn, kw = 0.13, 4, 10, 4, dict(anneal_stages=2, anneal_beta0=0.4)
    syn, _ = ctx.gen_syndromes(77, 0, n, L, p, like=torch.zeros(1, device="cuda"))
    opts = pkg.Opts(chains_per_class=R, n_sweeps=sweeps, burn_in=burn, lanes_per_bundle=lanes, **kw)
    cls, lz, mean = (x.cpu().numpy() for x in ctx.decode_ti(syn, L, p, opts, n_beta=n_beta, seed=31, id0=4))
    rows = syn.cpu().numpy()
    for i in (0, 1, n // 2, n - 1):
        k, rlz, rmean = O.decode_ti(L, p, 4, R, sweeps, 31, 4 + i, rows[i], n_beta=n_beta, burn_in=burn, **kw)
        assert int(cls[i]) == k
        assert (mean[i] == rmean).all() and (lz[i] == rlz).all()
    # few syndromes (other kernel, other streams) give the same numbers
    few = [x.cpu().numpy() for x in ctx.decode_ti(syn[:3], L, p, pkg.Opts(chains_per_class=R, n_sweeps=sweeps,
                                                                         burn_in=burn, **kw), n_beta=n_beta, seed=31,
                                                  id0=4)]
    for a, b in zip(few, (cls, lz, mean)):
        assert (a == b[:3]).all()


def _plan_case(pkg, ctx, Ls, p, opts, sw, seed, check):
    """A plan over fixed buffers, replayed on two inputs; items `check` against
    the oracle."""
    n = len(Ls)
    off = np.concatenate([[0], np.cumsum([2 * int(L) * (int(L) - 1) for L in Ls])])
    d_syn = torch.empty(int(off[-1]), dtype=torch.uint8, device="cuda")
    d_cls = torch.empty(n, dtype=torch.int32, device="cuda")
    d_sum = torch.empty((n, 4), dtype=torch.uint64, device="cuda")
    d_lr = torch.empty((n, 4), dtype=torch.float64, device="cuda")
    plan = pkg.RaggedPlan(ctx, Ls, p, d_syn, d_cls, d_sum, d_lr, opts=opts, n_sweeps=sw, seed=seed)
    for k in (0, 1, 0):
        rng = np.random.default_rng(900 + k)
        cat = (rng.random(int(off[-1])) < 0.2).astype(np.uint8)
        for i in check:
            cat[off[i]:off[i + 1]] = O.gen_syndromes(50 + k, i, 1, int(Ls[i]), p)[0][0]
        d_syn.copy_(torch.from_numpy(cat))
        plan.launch()
        torch.cuda.synchronize()
        cls, sums, lr = d_cls.cpu().numpy(), d_sum.cpu().numpy(), d_lr.cpu().numpy()
        for i in check:
            s = int(sw[i])
            burn = s * opts.burn_in // opts.n_sweeps
            akw = dict(anneal_stages=opts.anneal_stages, anneal_beta0=opts.anneal_beta0) if not opts.scan else {}
            ref = O.decode_one(int(Ls[i]), p, 4, opts.chains_per_class, s, seed, i, cat[off[i]:off[i + 1]],
                               burn_in=burn, scan=opts.scan, **akw)
            assert cls[i] == ref["cls"] and (sums[i] == ref["class_sum"]).all() and (lr[i] == ref["log_ratio"]).all()
    plan.close()


@pytest.mark.parametrize("R", [4, 9])
def test_plan_on_the_throughput_kernel(pkg, ctx, R):
    n = 1500
    Ls = np.random.default_rng(8).choice([5, 9, 13], size=n).astype(np.int32)
    sw = (Ls * 2).astype(np.uint32)
    opts = pkg.Opts(chains_per_class=R, n_sweeps=20, burn_in=8, anneal_stages=2, anneal_beta0=0.4)
    _plan_case(pkg, ctx, Ls, 0.14, opts, sw, 21, (0, 1, 2, 3, 4, 5, 6, 7, n // 2, n - 2, n - 1))


# more than 48 KiB of shared memory, the kernels' first use inside the capture
@pytest.mark.parametrize("scan", [0, 1])
def test_plan_with_large_shared_memory(pkg, ctx, scan):
    Ls = np.array([31, 28, 31], np.int32)
    sw = np.array([4, 3, 4], np.uint32)
    opts = pkg.Opts(chains_per_class=2, n_sweeps=4, burn_in=1, scan=scan)
    _plan_case(pkg, ctx, Ls, 0.12, opts, sw, 22, (0, 1, 2))
