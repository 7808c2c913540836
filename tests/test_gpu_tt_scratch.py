"""The scratch of weno_tt_round at many small problems: 20000 of them take at most 24 descriptor blocks of 400 bytes and
24 buffers of 1 KB, 0.69 GB."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_scratch_of_many_small_problems():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno as W
    build.build()
    count, rng = 20000, np.random.default_rng(3)
    x = [torch.from_numpy(rng.normal(size=s)).cuda() for s in ((3, 1, 1), (3, 1, 1), (3, 1, 1))]
    h = W.weno_init()
    W.weno_tt_round(h, [[(1.0, x), (1.0, x)]], 1e-9)  # (kernels and their local memory are loaded)
    problems = [[(1.0, x), (1.0, x)]] * count
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    outs = W.weno_tt_round(h, problems, 1e-9)
    W.weno_sync(h)
    took = before - torch.cuda.mem_get_info()[0] - torch.cuda.memory_reserved()
    assert took <= count * (24 * 400 + 24 * 1024), took
    G = [c.cpu().numpy() for c in outs[-1][0]]
    want = 2 * np.einsum("i,j,k->ijk", *[c.cpu().numpy().reshape(3) for c in x])
    got = np.einsum("ia,jab,kb->ijk", G[0][:, 0], G[1], G[2][:, :, 0])
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
    W.weno_destroy(h)
