"""The dense inverse of the coarsest matrix (blocked Gauss-Jordan whose rank-96 updates run on
the tensor cores as exact digit products), at the sizes where its blocks have remainders:
panels of 96 columns, sub-panels of 16, row tiles of 128, column tiles of 32, one and several
thread blocks of the panel's cluster, one and two rows of the panel per thread.

With block size 1 and one level, stage P alone is A^-1 applied to the right-hand side, so an
application must solve the system: the residual is held to n * 2^-53 times |A^-1| |A| with a
factor of 8 for the products and the decoupling scaling, and two such applications are equal
bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")


def _system(n, seed, small_diagonal):
    """Random sparse rows (the next index, 8 others, the diagonal); with a small diagonal the
    elimination has to exchange rows in almost every column."""
    rng = np.random.default_rng(seed)
    rp, ci, v = [0], [], []
    for i in range(n):
        c = np.unique(np.concatenate([[i, (i + 1) % n], rng.choice(n, min(n, 8), replace=False)]))
        x = rng.normal(size=c.size) * np.exp(rng.normal(size=c.size))
        if small_diagonal:
            x[c == i] *= 1e-3
            x[c == (i + 1) % n] += 5.0
        else:
            x[c == i] = 1.0 + np.abs(x[c != i]).sum()
        ci.append(c)
        v.append(x)
        rp.append(rp[-1] + c.size)
    return np.array(rp, np.int32), np.concatenate(ci).astype(np.int32), np.concatenate(v)


def _dense(rp, ci, v, n):
    a = np.zeros((n, n))
    a[np.repeat(np.arange(n), np.diff(rp)), ci] = v
    return a


@pytest.mark.parametrize("small_diagonal", [False, True])
@pytest.mark.parametrize("n", [1, 2, 15, 17, 95, 96, 97, 112, 128, 129, 191, 193, 300, 1025, 2111])
def test_inverse_solves_the_coarsest_system(n, small_diagonal):
    rp, ci, v = _system(n, n, small_diagonal)
    s = msp.Solver(n, 1, *(torch.from_numpy(x).to(DEV) for x in (rp, ci, v)), coarse_max=20000,
                   precond=msp.MSP_PREC_P_ONLY, colouring=msp.MSP_COLOURING_JP)
    assert s.num_levels == 1
    a = _dense(rp, ci, v, n)
    ainv = np.linalg.inv(a)
    bound = 8.0 * n * 2.0 ** -53 * np.linalg.norm(np.abs(ainv) @ np.abs(a), np.inf)
    rng = np.random.default_rng(5)
    for g in (rng.normal(size=n), np.eye(n)[n // 2], np.eye(n)[n - 1]):
        w = torch.empty(n, dtype=torch.float64, device=DEV)
        s.apply_precond(torch.from_numpy(g).to(DEV), w)
        x = w.cpu().numpy()
        ref = ainv @ g
        ref += ainv @ (g - a @ ref)
        assert np.abs(x - ref).max() <= bound * np.abs(ref).max(), np.abs(x - ref).max() / np.abs(ref).max()
        again = torch.empty_like(w)
        s.apply_precond(torch.from_numpy(g).to(DEV), again)
        assert torch.equal(w, again)
    s.close()


def test_two_rows_of_the_panel_per_thread():
    """More than 8,192 rows: narrower sub-panels, two rows per thread."""
    n = 8300
    rp, ci, v = _system(n, 1, True)
    s = msp.Solver(n, 1, *(torch.from_numpy(x).to(DEV) for x in (rp, ci, v)), coarse_max=20000,
                   precond=msp.MSP_PREC_P_ONLY, colouring=msp.MSP_COLOURING_JP)
    a = torch.from_numpy(_dense(rp, ci, v, n)).to(DEV)
    g = torch.from_numpy(np.random.default_rng(2).normal(size=n)).to(DEV)
    w = torch.empty_like(g)
    s.apply_precond(g, w)
    ref = torch.linalg.solve(a, g)
    # torch's own solve differs from the exact solution by as much: twice the bound of one
    cond = float(torch.linalg.norm(torch.linalg.inv(a), float("inf")) * torch.linalg.norm(a, float("inf")))
    assert float((w - ref).abs().max() / ref.abs().max()) <= 2 * 8.0 * n * 2.0 ** -53 * cond
    s.close()


def test_singular_coarsest_matrix_is_reported():
    n = 130
    rp, ci, v = _system(n, 3, False)
    a = _dense(rp, ci, v, n)
    a[100] = 0.0
    a[100, 99], a[100, 100] = a[99, 99], a[99, 100]  # row 100 = row 99's two leading entries
    a[99] = 0.0
    a[99, 99], a[99, 100] = a[100, 99], a[100, 100]
    a[99, 100] = a[100, 100] = 1.0
    a[99, 99] = a[100, 99] = 1.0
    rows, cols = np.nonzero(a)
    rp = np.searchsorted(rows, np.arange(n + 1)).astype(np.int32)
    with pytest.raises(msp.MspError) as e:
        msp.Solver(n, 1, torch.from_numpy(rp).to(DEV), torch.from_numpy(cols.astype(np.int32)).to(DEV),
                   torch.from_numpy(a[rows, cols]).to(DEV), coarse_max=20000, colouring=msp.MSP_COLOURING_JP)
    assert e.value.status == msp._native.MSP_ERR_SINGULAR_BLOCK
