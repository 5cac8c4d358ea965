"""VerticesGrouping on the GPU takes several frontier vertices per round; its colours must be
those of one pick at a time (the oracle), on graphs where the rounds can go wrong: dense
second circles past the lists' hash table and past the entries kept in registers, hubs joined
to many vertices, several components (picks by label), sizes around the groups of 32 and 1024
labels, and vertices without neighbours."""
import numpy as np
import pytest

import oracle
from synthetic.jacobian import BSRMatrix

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")


def _matrix(n, edges):
    """Diagonally dominant scalar matrix with the symmetric pattern of the edges."""
    e = np.array(sorted({(min(a, b), max(a, b)) for a, b in edges if a != b}), np.int64).reshape(-1, 2)
    rows = np.concatenate([e[:, 0], e[:, 1], np.arange(n)])
    cols = np.concatenate([e[:, 1], e[:, 0], np.arange(n)])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    deg = np.bincount(rows, minlength=n)
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(deg, out=rp[1:])
    v = np.where(rows == cols, deg[rows].astype(float), -1.0).reshape(-1, 1, 1)
    return BSRMatrix(n, 1, rp, cols.astype(np.int32), v, n, 0, (n, 1, 1))


def _random(n, per, seed):
    rng = np.random.default_rng(seed)
    return [(i, int(j)) for i in range(n) for j in rng.integers(0, n, per)]


def _near(n, reach, per, seed):
    rng = np.random.default_rng(seed)
    return [(i, int(j)) for i in range(n) for j in np.clip(i + rng.integers(-reach, reach + 1, per), 0, n - 1)]


GRAPHS = {
    "single": lambda: (1, []),
    "isolated": lambda: (70, []),
    "path_33": lambda: (33, [(i, i + 1) for i in range(32)]),
    "grid_1023": lambda: (1023, [(i, i + 1) for i in range(1022)] + [(i, i + 31) for i in range(992)]),
    "grid_1025": lambda: (1025, [(i, i + 1) for i in range(1024)] + [(i, i + 25) for i in range(1000)]),
    "components": lambda: (3000, [(i, i + 1) for i in range(2999) if i % 10 != 9]),
    "near_4000": lambda: (4000, _near(4000, 40, 6, 1)),
    "random_2500": lambda: (2500, _random(2500, 4, 2)),
    "dense_circles": lambda: (900, _near(900, 30, 24, 3)),      # second circles over 128 entries
    "past_the_table": lambda: (700, _random(700, 16, 4)),       # raw second circles over 384
    "hub": lambda: (1500, [(0, i) for i in range(1, 1500)] + _near(1500, 5, 2, 5)),
    "cliques": lambda: (600, [(20 * c + a, 20 * c + b) for c in range(30) for a in range(20) for b in range(a)]
                        + [(20 * c, 20 * c + 20) for c in range(29)]),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_colours_equal_the_sequential_ones(name):
    n, edges = GRAPHS[name]()
    a = _matrix(n, edges)
    s = msp.Solver(a.nb, a.b, *(torch.from_numpy(x).to(DEV) for x in
                                (a.row_ptr, a.col_idx, a.values.reshape(-1))), coarse_max=20000)
    colour, g = s.colour0()
    s.close()
    o = oracle.Oracle(a, coarse_max=20000)
    ref, gref = o.colour0()
    assert g == gref
    assert np.array_equal(colour, ref)
