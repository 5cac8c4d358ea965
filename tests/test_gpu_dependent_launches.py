"""Colour classes launched as programmatic dependents read what earlier classes wrote only after
their wait, and not through the read-only path.  Small grids whose classes hold both well rows
of more than 16 blocks and cells (stage N, one thread block per well row beside the cells'
threads): a stage-N application of several sweeps within 1e-10 of the oracle, and 50 more of
other vectors interleaved with it equal bit for bit, in FP64 and in FP32.  And grids of stars, whose
first class holds long rows only (stage R: the class that follows the kernel that writes its
right-hand side)."""
import numpy as np
import pytest

import oracle
from synthetic import box_jacobian
from synthetic.jacobian import BSRMatrix

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")
LONG = 16  # blocks of a row above which a thread block takes it


def _vec(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _check(a, o, cfg):
    rng = np.random.default_rng(a.b)
    xs = [rng.normal(size=a.n) for _ in range(2)]
    ref = o.apply_precond(xs[0])
    for precision in (msp.MSP_PRECISION_FP64, msp.MSP_PRECISION_FP32):
        g = msp.Solver(a.nb, a.b, _vec(a.row_ptr), _vec(a.col_idx), _vec(a.values.reshape(-1)),
                       precision=precision, **cfg)
        xd = [_vec(x) for x in xs]
        first, w = torch.empty_like(xd[0]), torch.empty_like(xd[0])
        g.apply_precond(xd[0], first)
        if precision == msp.MSP_PRECISION_FP64:
            assert np.abs(first.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        for _ in range(50):  # values of the other vector in between: nothing of them may stay
            g.apply_precond(xd[1], w)
            g.apply_precond(xd[0], w)
            assert torch.equal(w, first)
        g.close()


@pytest.mark.parametrize("b", [2, 3, 5, 8])
def test_classes_of_well_rows_and_cells(b):
    a = box_jacobian(13, 5, 30, b, 2, layered=True, kz_ratio=0.1, n_wells=4)
    cfg = dict(coarse_max=80, precond=msp.MSP_PREC_N_ONLY, bgs_sweeps=8)
    o = oracle.Oracle(a, **cfg)
    colour, g = o.colour0()
    long = np.diff(a.row_ptr) > LONG
    counts = [(int((colour == c).sum()), int(((colour == c) & long).sum())) for c in range(1, g + 1)]
    assert sum(0 < nl < n and n * (b - 1) <= 8192 for n, nl in counts) >= 1, counts
    _check(a, o, cfg)
    o.close()


def _stars(hubs, leaves, b):
    """Disjoint stars: the hubs (rows of leaves + 1 blocks) have the largest degree, and no
    second circle joins the frontier before them."""
    n = hubs * (leaves + 1)
    rng = np.random.default_rng(hubs)
    rp, ci, v = [0], [], []
    for h in range(hubs):
        base = h * (leaves + 1)
        for i in range(leaves + 1):
            cols = range(base, base + leaves + 1) if i == 0 else (base, base + i)
            for c in cols:
                ci.append(c)
                blk = 0.1 * rng.normal(size=(b, b)) / leaves
                v.append(blk + np.eye(b) if c == base + i else blk)
            rp.append(len(ci))
    return BSRMatrix(n, b, np.array(rp, np.int32), np.array(ci, np.int32), np.array(v), n, 0, (n, 1, 1))


@pytest.mark.parametrize("precond", [msp.MSP_PREC_R_ONLY, msp.MSP_PREC_MSP])
@pytest.mark.parametrize("b", [1, 4, 7])
def test_first_class_of_long_rows_only(b, precond):
    a = _stars(6, 40, b)
    cfg = dict(coarse_max=400, precond=precond)
    o = oracle.Oracle(a, **cfg)
    colour, g = o.colour0()
    assert (np.diff(a.row_ptr)[colour == 1] > LONG).all() and g == 2
    _check(a, o, cfg)
    o.close()
