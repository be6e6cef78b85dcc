"""Start frames at the edges of the kernel's split (8, 16 or 32 lanes per
syndrome, so 4, 2 or 1 syndromes per warp) against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_2669_gb300 import build as b
    b.build()
    import paper_1302_2669_gb300 as P
    c = P.Context(0)
    yield c
    c.close()


# the last warp of a launch with one to all of its syndromes, the last block
# with one to all of its warps
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 15, 17, 33])
@pytest.mark.parametrize("L", [2, 7, 8, 9, 16, 17, 31])
def test_start_frames_edges(ctx, L, n):
    rng = np.random.default_rng(100 * L + n)
    syn = (rng.random((n, O.nstab(L))) < rng.random((n, 1))).astype(np.uint8)
    syn[-1] = 1
    # rows past the end must not be written
    frames = torch.full((n + 4, 2, O.words(L)), 0x5A5A5A5A, dtype=torch.int32, device="cuda").view(torch.uint32)
    code = torch.full((n + 4,), 77, dtype=torch.int32, device="cuda")
    ctx.start_frames(torch.from_numpy(syn).cuda(), L, frames=frames, e0_class=code)
    torch.cuda.synchronize()
    fr, code = frames.cpu().numpy(), code.cpu().numpy()
    for i in range(n):
        ex, ez = O.pure_error(L, syn[i])
        assert (fr[i, 0] == O.pack_bits(ex)).all() and (fr[i, 1] == O.pack_bits(ez)).all()
        assert code[i] == O.class_code(L, ex, ez)
    assert (fr[n:] == 0x5A5A5A5A).all() and (code[n:] == 77).all()
