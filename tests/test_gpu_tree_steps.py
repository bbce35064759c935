"""Tree passes over the byte maps against the oracle where they can go wrong:
levels whose rows hold fewer than 16 cells, exactly 16, and several 16-cell
steps; periodic and reflecting walls mixed per direction (a step's neighbours
wrap, or stop at the wall); remeshes of every depth inside a macro step (the
frozen-level test of refinements); a chunk border inside a level."""
import numpy as np
import pytest

import oracle
from paper_1905_08717_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_08717_gb300 import build
    build.build()


def _data(dim, L, seed):
    """a rough field: a few waves plus a step, so that leaves of every level meet every wall"""
    rng = np.random.default_rng(seed)
    n = 1 << L
    x = (np.arange(n) + 0.5) / n
    g = np.meshgrid(*([x] * dim), indexing="ij")
    u = np.zeros((n,) * dim)
    for _ in range(3):
        k = rng.integers(1, 4, dim)
        u += rng.normal() * np.sin(sum(2 * np.pi * kk * gg for kk, gg in zip(k, g)) + rng.uniform(0, 6.28))
    r2 = sum((gg - rng.uniform(0, 1)) ** 2 for gg in g)
    return (0.3 * u + (r2 < 0.05))[None].copy()


P, N, D = I.BC_PERIODIC, I.BC_NEUMANN, I.BC_DIRICHLET0


@pytest.mark.parametrize("dim,L,lb,bc,mode", [
    (1, 3, 1, (P, P, P), I.TIME_LT), (1, 4, 2, (N, N, N), I.TIME_LT), (1, 5, 2, (D, D, D), I.TIME_LT),
    (1, 9, 0, (P, P, P), I.TIME_LT), (1, 13, 6, (N, N, N), I.TIME_LT),
    (2, 4, 1, (P, N, P), I.TIME_LT), (2, 5, 2, (N, P, P), I.TIME_LT), (2, 6, 3, (P, P, P), I.TIME_LT),
    (2, 7, 2, (D, P, P), I.TIME_LT), (2, 6, 2, (P, D, P), I.TIME_GTS),
    (3, 4, 1, (P, N, D), I.TIME_LT), (3, 5, 2, (N, P, P), I.TIME_LT), (3, 5, 1, (P, P, P), I.TIME_GTS),
])
def test_trees_equal_the_oracle(dim, L, lb, bc, mode):
    import paper_1905_08717_gb300 as pkg
    p = I.Problem(dim=dim, equation=I.EQ_BURGERS, max_level=L, min_level=lb, eps=0.1 if dim == 3 else 2e-2, time_mode=mode, bc=bc)
    q = _data(dim, L, 7 * dim + L)
    g, o = pkg.Solver(p, q), oracle.Oracle(p, q)
    t = 6.0 / (1 << L)
    for k in (1, 2, 3):
        g.step(k * t)
        o.step(k * t)
        kg, vg = g.leaves()
        ko, vo = o.leaves()
        assert np.array_equal(kg, ko), f"leaf sets differ at {k}"
        assert np.abs(vg - vo).max() <= 1e-12 * np.abs(vo).max()
    g.close()
