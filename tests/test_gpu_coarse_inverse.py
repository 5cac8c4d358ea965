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


def _grid(nx, ny, nz, sigma, seed):
    """7-point matrix with lognormal permeability exp(sigma N), rows with unit diagonals."""
    rng = np.random.default_rng(seed)
    n = nx * ny * nz
    k = np.exp(sigma * rng.normal(size=(nz, ny, nx)))
    idx, a = np.arange(n).reshape(nz, ny, nx), np.zeros((n, n))
    for ax in range(3):
        i, kk = np.moveaxis(idx, ax, 0), np.moveaxis(k, ax, 0)
        t = (2 * kk[1:] * kk[:-1] / (kk[1:] + kk[:-1])).ravel()
        a[i[1:].ravel(), i[:-1].ravel()] = -t * rng.uniform(0.1, 1, t.size)
        a[i[:-1].ravel(), i[1:].ravel()] = -t * rng.uniform(0.1, 1, t.size)
    a[np.arange(n), np.arange(n)] = rng.uniform(0.5, 2.0, n) - a.sum(1)
    return a / np.diag(a)[:, None]


SCALES = {  # binary exponents of the rows and of the columns
    "unit": lambda rng, n: (np.zeros(n, int), np.zeros(n, int)),
    "last_rows_up": lambda rng, n: (np.where(np.arange(n) >= n - 4, 33, 0), np.zeros(n, int)),
    "last_rows_down": lambda rng, n: (np.where(np.arange(n) >= n - 4, -33, 0), np.zeros(n, int)),
    "first_rows_up": lambda rng, n: (np.where(np.arange(n) < 3, 47, 0), np.zeros(n, int)),
    "last_unknowns": lambda rng, n: (np.zeros(n, int), np.where(np.arange(n) >= n - 4, -33, 0)),
    "rows": lambda rng, n: (rng.integers(-30, 31, n), np.zeros(n, int)),
    "columns": lambda rng, n: (np.zeros(n, int), rng.integers(-30, 31, n)),
    "both": lambda rng, n: (rng.integers(-30, 31, n), rng.integers(-30, 31, n)),
    "tiny": lambda rng, n: (np.full(n, -900), np.zeros(n, int)),
    "huge": lambda rng, n: (np.full(n, 900), np.zeros(n, int)),
}


@pytest.mark.parametrize("scale", sorted(SCALES))
@pytest.mark.parametrize("matrix", ["grid", "spread_grid", "exchanges"])
def test_rows_and_columns_in_other_units(matrix, scale):
    """Without the decoupling weights the coarsest rows keep the units of the caller's rows.
    A = 2^r A0 2^c has the inverse 2^-c A0^-1 2^-r exactly, and elimination in FP64 keeps
    |E| <= n 2^-53 |A^-1| |A| |A^-1| entry by entry (times a small factor) for all of them, as
    does one step of refinement in the working precision: the same bound, with a factor of 8
    for the inverse and 8 for the reference (an FP64 inverse of A0 and such a step), for whole
    vectors and for single columns of the inverse, whose entries span ten orders of magnitude."""
    if matrix == "exchanges":
        a0 = _dense(*_system(300, 7, True), 300)
    else:
        a0 = _grid(8, 7, 6, 4.0 if matrix == "spread_grid" else 1.0, 3)
    n = len(a0)
    rng = np.random.default_rng(11)
    r, c = SCALES[scale](rng, n)
    a = np.ldexp(np.ldexp(a0, r[:, None]), c[None, :])
    x0 = np.linalg.inv(a0)
    x0 += x0 @ (np.eye(n) - a0 @ x0)
    bound = 16.0 * n * 2.0 ** -53 * (np.abs(x0) @ np.abs(a0) @ np.abs(x0))
    rows, cols = np.nonzero(a)
    rp = np.searchsorted(rows, np.arange(n + 1)).astype(np.int32)
    s = msp.Solver(n, 1, *(torch.from_numpy(x).to(DEV) for x in (rp, cols.astype(np.int32), a[rows, cols])),
                   coarse_max=20000, precond=msp.MSP_PREC_P_ONLY, colouring=msp.MSP_COLOURING_JP, decoupling=0)
    assert s.num_levels == 1
    for g in [rng.normal(size=n)] + [np.eye(n)[j] for j in (0, n // 2, n - 5, n - 1)]:
        w = torch.empty(n, dtype=torch.float64, device=DEV)
        s.apply_precond(torch.from_numpy(np.ldexp(g, r)).to(DEV), w)
        x = np.ldexp(w.cpu().numpy(), c)
        assert (np.abs(x - x0 @ g) <= bound @ np.abs(g)).all()
    s.close()
