"""Krylov kernels at the sizes where their loops have remainders: vectors of fewer elements than
a block and just past the two-elements-a-thread and four-in-flight strides, bases of 1 to 33
vectors (groups of 8, 9, 17, ... dot products), batches whose chunks end inside a block's
stride.  A solve of restart 32 must satisfy its tolerance and its Arnoldi estimate must agree
with the true residual, which fails when a dot product or an update misses an element."""
import numpy as np
import pytest

from synthetic import box_jacobian, random_rhs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


@pytest.mark.parametrize("restart", [1, 7, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("dims,b", [((2, 2, 2), 1), ((5, 5, 5), 2), ((8, 8, 8), 1), ((9, 19, 3), 1),
                                    ((16, 16, 4), 1), ((11, 10, 7), 2), ((23, 19, 13), 3)])
def test_estimate_and_true_residual_agree(dims, b, restart):
    a = box_jacobian(*dims, b, 3, layered=True, kz_ratio=0.1)
    s = msp.Solver(a.nb, b, _dev(a.row_ptr), _dev(a.col_idx), _dev(a.values.reshape(-1)), coarse_max=20,
                   restart=restart, precond=msp.MSP_PREC_R_ONLY, max_it=33)
    rhs = random_rhs(a, 5)
    x = torch.zeros(a.n, dtype=torch.float64, device=DEV)
    info = s.solve(_dev(rhs), x, 1e-10)
    r = rhs - a.to_scipy() @ x.cpu().numpy()
    true = np.linalg.norm(r) / np.linalg.norm(rhs)
    # both from FP64 sums of n terms; the residual itself is formed with errors of
    # n eps |A| |x| / |b|
    slack = 4 * a.n * 2.0 ** -53 * np.linalg.norm(abs(a.to_scipy()) @ np.abs(x.cpu().numpy())) / np.linalg.norm(rhs)
    assert abs(info["rel_residual"] - true) <= slack + 1e-12 * true
    assert abs(info["rel_residual_est"] - true) <= slack + 1e-6 * true, (info, true)
    s.close()


@pytest.mark.parametrize("count", [1, 3, 40])
def test_batch_chunks_with_remainders(count):
    ms = [box_jacobian(5 + i % 4, 6 + i % 3, 7 + i % 5, 3, 10 + i, layered=True, kz_ratio=0.1,
                       n_wells=i % 2) for i in range(count)]
    nb, b, rp, ci, v, off = msp.stack_block_diagonal(ms)
    s = msp.BatchSolver(nb, b, _dev(rp), _dev(ci), _dev(v), off, coarse_max=60)
    rhs = np.concatenate([random_rhs(m, 20 + i) for i, m in enumerate(ms)])
    x = torch.zeros(nb * b, dtype=torch.float64, device=DEV)
    infos = s.solve_batch(_dev(rhs), x, 1e-9)
    xs = x.cpu().numpy()
    for i, m in enumerate(ms):
        lo, hi = off[i] * b, off[i + 1] * b
        rel = np.linalg.norm(rhs[lo:hi] - m.to_scipy() @ xs[lo:hi]) / np.linalg.norm(rhs[lo:hi])
        assert infos[i]["status"] == 0 and rel <= 1.001e-9, (i, infos[i], rel)
    s.close()
