"""The residual restriction of an AMG level of more than 262,144 rows reads only the entries right
of the diagonal (after one forward colour sweep from zero the others cancel).  On a level-0
matrix just above that size, with well rows that are longer than the ELL copy (taken from the CSR
form): the application of stage P alone and of the whole preconditioner within 1e-10 of the oracle,
the solve within one iteration of the oracle's in FP64 and with the FP32 preconditioner; and with
two forward sweeps, where the whole rows are read."""
import numpy as np
import pytest

import oracle
from synthetic import box_jacobian, random_rhs

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")


def _vec(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _solver(a, **cfg):
    return msp.Solver(a.nb, a.b, _vec(a.row_ptr), _vec(a.col_idx), _vec(a.values.reshape(-1)), **cfg)


@pytest.mark.parametrize("pre_sweeps,b,precond", [(1, 1, msp.MSP_PREC_P_ONLY), (1, 2, msp.MSP_PREC_MSP),
                                                  (2, 1, msp.MSP_PREC_P_ONLY)])
def test_level_of_more_than_262144_rows(pre_sweeps, b, precond):
    a = box_jacobian(65, 65, 63, b, 9, layered=True, kz_ratio=0.1, n_wells=3)
    assert a.nb > 262144 and int((np.diff(a.row_ptr) - 1 > 32).sum()) == 3
    cfg = dict(coarse_max=1500, precond=precond, pre_sweeps=pre_sweeps, colouring=msp.MSP_COLOURING_JP)
    g, o = _solver(a, **cfg), oracle.Oracle(a, **cfg)
    for seed in (1, 2):
        x = random_rhs(a, seed)
        w = torch.zeros(a.n, dtype=torch.float64, device=DEV)
        g.apply_precond(_vec(x), w)
        ref = o.apply_precond(x)
        assert np.abs(w.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    rhs = random_rhs(a, 3)
    _, io = o.solve(rhs, 1e-6)
    for precision in (msp.MSP_PRECISION_FP64, msp.MSP_PRECISION_FP32):
        s = g if precision == msp.MSP_PRECISION_FP64 else _solver(a, precision=precision, **cfg)
        x = torch.zeros(a.n, dtype=torch.float64, device=DEV)
        info = s.solve(_vec(rhs), x, 1e-6)
        assert info["status"] == io["status"] == 0 and abs(info["iterations"] - io["iterations"]) <= 1, (info, io)
        assert np.linalg.norm(rhs - a.to_scipy() @ x.cpu().numpy()) <= 1.001e-6 * np.linalg.norm(rhs)
        s.close()
    o.close()
