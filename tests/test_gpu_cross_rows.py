"""weno_tt_cross refuses fiber matrices of more rows than maxvol's row masks hold (65536), before any launch, and takes
the largest that they do."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ranks,fits", [((4, 1025, 14), (4, 64), False),
                                          ((64, 1025, 14), (64, 4), False), ((65537, 4, 4), (2, 2), False),
                                          ((65536, 4, 4), (2, 2), True), ((4, 4, 13108), (2, 2), False)])
def test_rows_of_the_fiber_matrices(n, ranks, fits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno as W
    build.build()
    rng = np.random.default_rng(1)
    r = (3, 3)
    cores = []
    for mean in (1.0, 0.3, 0.2, 0.1, 2.6):
        g = [0.1 * rng.normal(size=s) for s in ((n[0], 1, r[0]), (n[1], r[0], r[1]), (n[2], r[1], 1))]
        for m in range(3):
            g[m][:, 0, 0] = mean if m == 0 else 1.0
        cores.append([torch.from_numpy(x.astype(np.float32)).cuda() for x in g])
    inst = dict(n=n, r=r, cores=cores, h=[1.0 / k for k in n], bc=((0, 0),) * 3, alpha=2.0)
    J1 = torch.from_numpy(np.stack([rng.permutation(max(n[1], ranks[0]))[:ranks[0]] % n[1], rng.integers(0, n[2], ranks[0]),
                                    np.arange(ranks[0]) % 5], 1).astype(np.int32)).cuda()
    k = rng.permutation(5 * n[2])[:ranks[1]]
    J2 = torch.from_numpy(np.stack([k // 5, k % 5], 1).astype(np.int32)).cuda()
    h = W.weno_init()
    if fits:
        (o,) = W.weno_tt_cross(h, [inst], 0, [ranks], [J1], [J2], sweeps=0, fp64_check=True)
        W.weno_sync(h)
        assert all(bool(torch.isfinite(c).all()) for c in o["cores"])
    else:
        with pytest.raises(W.WenoError, match="status 5"):
            W.weno_tt_cross(h, [inst], 0, [ranks], [J1], [J2], sweeps=0, fp64_check=True)
    W.weno_destroy(h)
