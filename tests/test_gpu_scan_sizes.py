"""Random scan at the ends of its range (smallest and largest codes, planes of
4 to 32 chains with partly filled bundles, every noise model, both codes)
against the oracle, bit for bit."""
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


@pytest.mark.parametrize("toric,L,R,n", [(0, 2, 1, 9), (0, 3, 9, 2), (0, 16, 3, 3), (0, 31, 2, 2), (1, 2, 1, 3),
                                         (1, 4, 3, 2), (1, 30, 1, 1)])
@pytest.mark.parametrize("noise", [0, 1, 2])
def test_scan_at_the_ends_of_its_range(pkg, ctx, toric, L, R, n, noise):
    p, sweeps, burn, e = 0.1, 3, 1, (3, 1, 2)
    K = 16 if toric else 4
    syn = (O.t_gen_syndromes if toric else O.gen_syndromes)(5100 + L, 0, n, L, p)[0]
    opts = pkg.Opts(n_classes=K, chains_per_class=R, n_sweeps=sweeps, burn_in=burn, scan=1, noise=noise,
                    pauli_energy=e if noise == 2 else (1, 1, 1))
    out = ctx.decode_ex(torch.from_numpy(syn).cuda(), L, p, opts, seed=17, id0=2, accepts=True)
    for i in range(n):
        ref = O.decode_one(L, p, K, R, sweeps, 17, 2 + i, syn[i], burn_in=burn, scan=1, noise=noise,
                           energy=e if noise == 2 else None, accepts=True)
        assert int(out["cls"][i]) == ref["cls"]
        for k in ("class_sum", "log_ratio", "chain_sum", "chain_n", "accepts"):
            assert (out[k][i].cpu().numpy() == ref[k]).all(), k
        fr = out["chain_frames"][i].cpu().numpy()
        assert (fr[:, 0, :] == O.pack_bits(ref["frames_x"])).all()
        assert (fr[:, 1, :] == O.pack_bits(ref["frames_z"])).all()


# the last round of a colour partly filled or not, one bundle or many: the
# rule's lane split against fixed ones
@pytest.mark.parametrize("L,R,n", [(5, 4, 5000), (9, 4, 9000), (13, 8, 1500), (22, 4, 1300)])
def test_lane_rule_does_not_change_results(pkg, ctx, L, R, n):
    syn, _ = ctx.gen_syndromes(61 + L, 0, n, L, 0.12, like=torch.zeros(1, device="cuda"))
    runs = []
    for lam in (0, 8, 16, 32):
        o = pkg.Opts(chains_per_class=R, n_sweeps=6, burn_in=2, lanes_per_bundle=lam)
        try:
            runs.append(ctx.decode(syn, L, 0.12, o, seed=23))
        except pkg.SurfmcmcError:
            assert lam == 8      # more shared memory than a block may use
    for r in runs[1:]:
        for a, b in zip(runs[0], r):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert len(runs) >= 3
