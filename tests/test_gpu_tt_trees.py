"""TT-rounding where its QR trees and the clustered SVD can go wrong: many row chunks and levels, one sub-block, the
largest summed ranks on one CTA and on several, batches large enough for one CTA per SVD, exactly dependent terms,
zero terms, values far from 1.  Checked on the full tensor: ||X - Y|| <= (eps + 1e-13) ||X|| (1e-13: 64 FP64 roundings
of the largest entries on either side), ||X|| itself to 1e-13, and left-orthonormal first and middle cores to 1e-12
(the SVD's columns count as orthogonal from a cosine of 8 * 96 * 2^-52 = 1.7e-13, a few of which add up in a Gram
entry's row)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno
    build.build()
    weno.lib()
    return weno


def tt(rng, n, r, decay=0.0, scale=1.0):
    g = [rng.normal(size=(n[0], 1, r[0])), rng.normal(size=(n[1], r[0], r[1])), rng.normal(size=(n[2], r[1], 1))]
    g[1] *= 10.0 ** (-decay * (np.arange(r[0])[:, None] / r[0] + np.arange(r[1])[None] / r[1]))
    g[0] *= scale
    return g


def full(g):
    return np.einsum("ia,jab,kb->ijk", g[0][:, 0], g[1], g[2][:, :, 0], optimize=True)


def check(W, problems, eps):
    h = W.weno_init()
    outs = W.weno_tt_round(h, [[(c, [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in g]) for c, g in t]
                               for t in problems], eps)
    W.weno_sync(h)
    for terms, (cores, norm) in zip(problems, outs):
        X = sum(c * full(g) for c, g in terms)
        G = [c.cpu().numpy() for c in cores]
        size = np.linalg.norm(X)
        terms_size = max(abs(c) * np.linalg.norm(full(g)) for c, g in terms)
        assert np.linalg.norm(full(G) - X) <= eps * size + 1e-13 * terms_size
        assert abs(norm - size) <= 1e-13 * terms_size
        a = G[0][:, 0]
        b = G[1].transpose(1, 0, 2).reshape(-1, G[1].shape[2])
        for m in (a, b):
            assert np.abs(m.T @ m - np.eye(m.shape[1])).max() <= 1e-12
    W.weno_destroy(h)
    return outs


@pytest.mark.parametrize("n,ranks,decay", [
    ((40, 200, 96), [(32, 32), (16, 32)], 3.0),      # 80 sub-blocks of 96 rows in the middle QR
    ((30, 100, 33), [(3, 2)], 0.0),
    ((97, 50, 100), [(32, 32), (32, 32), (32, 32)], 4.0),   # summed ranks 96 everywhere
    ((89, 40, 90), [(30, 30), (30, 30), (29, 29)], 4.0),    # 89: one past a single CTA
    ((1, 9, 7), [(1, 2), (1, 3)], 0.0),
    ((2, 1, 2), [(1, 1)], 0.0),
])
@pytest.mark.parametrize("eps", [1e-12, 1e-4])
def test_sums(W, n, ranks, decay, eps):
    rng = np.random.default_rng(sum(n))
    check(W, [[(rng.uniform(0.5, 2), tt(rng, n, r, decay)) for r in ranks]], eps)


def test_batch_on_one_cta_each(W):
    rng = np.random.default_rng(5)
    problems = []
    for k in range(160):
        n = tuple(int(v) for v in rng.integers(3, 40, 3))
        problems.append([(1.0, tt(rng, n, rng.integers(1, 8, 2), 2.0)), (0.1, tt(rng, n, rng.integers(1, 8, 2), 2.0))])
    check(W, problems, 1e-9)


@pytest.mark.parametrize("scale", [1e-90, 1.0, 1e90])
def test_dependent_and_zero_terms(W, scale):
    rng = np.random.default_rng(6)
    n = (33, 24, 40)
    x = tt(rng, n, (12, 10), 3.0, scale)
    z = [np.zeros_like(g) for g in x]
    (G, _), (H, _), _, (K, _) = check(W, [[(1.0, x), (1e-3, x)], [(1.0, x), (-0.5, x), (2.0, z)], [(1.0, z), (2.0, z)],
                                          [(1.0, x), (1e-9, tt(rng, n, (4, 4), 0.0, scale))]], 1e-12)
    assert (G[0].shape[2], G[1].shape[2]) == (12, 10) and (H[0].shape[2], H[1].shape[2]) == (12, 10)
    assert (K[0].shape[2], K[1].shape[2]) == (16, 14)


def test_eps_zero_keeps_an_orthonormal_basis(W):
    rng = np.random.default_rng(7)
    x = tt(rng, (20, 11, 15), (5, 4), 1.0)
    check(W, [[(1.0, x), (1.0, x)], [(1.0, x)]], 0.0)
