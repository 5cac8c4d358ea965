"""The panels' LU of the coarsest inverse in the variants that a whole GPU takes only for very
large matrices, or not at all: more rows of the panel per thread (1, 2, 4, 16, 32, with narrower
sub-panels) and clusters of 8 thread blocks (what is portable) and 16.  The inverse is held to
n * 2^-53 |A^-1| |A| |A^-1| entry by entry with a factor of 8, the NumPy reference (refined once)
to another 8; and a matrix of more than 16,384 rows by its residual."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2208_08594_gb300 import _native  # noqa: E402

DEV = torch.device("cuda:0")


def _system(n, seed):
    """Random sparse rows whose elimination has to exchange rows in almost every column."""
    rng = np.random.default_rng(seed)
    rp, ci, v = [0], [], []
    for i in range(n):
        c = np.unique(np.concatenate([[i, (i + 1) % n], rng.integers(0, n, 8)]))
        x = rng.normal(size=c.size) * np.exp(rng.normal(size=c.size))
        x[c == i] *= 1e-3
        x[c == (i + 1) % n] += 5.0
        ci.append(c)
        v.append(x)
        rp.append(rp[-1] + c.size)
    return np.array(rp, np.int32), np.concatenate(ci).astype(np.int32), np.concatenate(v)


def _inverse(rp, ci, v, cluster, panel_rows, wait_ns=-1, status=_native.MSP_OK):
    n = len(rp) - 1
    d = [torch.from_numpy(x).to(DEV) for x in (rp, ci, v)]
    out = torch.empty(n, n, dtype=torch.float64, device=DEV)
    st = _native.lib().msp_test_inverse(C.c_int32(n), C.c_int32(len(ci)), *(C.c_void_p(x.data_ptr()) for x in d),
                                        C.c_void_p(out.data_ptr()), C.c_int32(cluster), C.c_int32(panel_rows),
                                        C.c_int64(wait_ns), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == status, st
    return out


@pytest.mark.parametrize("cluster", [8, 16])
@pytest.mark.parametrize("panel_rows", [1, 2, 4, 16, 32])
@pytest.mark.parametrize("n", [1, 97, 700, 2111])
def test_rows_per_thread_and_cluster_size(n, panel_rows, cluster):
    rp, ci, v = _system(n, n)
    a = np.zeros((n, n))
    a[np.repeat(np.arange(n), np.diff(rp)), ci] = v
    x0 = np.linalg.inv(a)
    x0 += x0 @ (np.eye(n) - a @ x0)
    bound = 16.0 * n * 2.0 ** -53 * (np.abs(x0) @ np.abs(a) @ np.abs(x0))
    assert (np.abs(_inverse(rp, ci, v, cluster, panel_rows).cpu().numpy() - x0) <= bound).all()


@pytest.mark.parametrize("n,cluster", [(4500, 8), (16500, 0)])
def test_more_rows_than_one_per_thread(n, cluster):
    """Two rows a thread on 8 blocks, four on 16 (the device's choice): the residual of two
    columns and a vector, n 2^-53 |A| |A^-1| |A| |A^-1| |g| with a factor of 8."""
    rp, ci, v = _system(n, 3)
    x = _inverse(rp, ci, v, cluster, 0)
    rows = torch.from_numpy(np.repeat(np.arange(n), np.diff(rp))).to(DEV)
    cols, vals = torch.from_numpy(ci).to(DEV).long(), torch.from_numpy(v).to(DEV)

    def product(w, y):  # sparse matrix with values w, times y
        return torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, w * y[cols])

    g = torch.zeros(3, n, dtype=torch.float64, device=DEV)
    g[0] = torch.from_numpy(np.random.default_rng(2).normal(size=n)).to(DEV)
    g[1, n // 2] = g[2, n - 1] = 1.0
    for gi in g:
        ag = product(vals.abs(), x.abs() @ product(vals.abs(), x.abs() @ gi.abs()))
        r = gi - product(vals, x @ gi)
        assert bool((r.abs() <= 8.0 * n * 2.0 ** -53 * ag).all())


@pytest.mark.parametrize("n", [1, 97, 2111])
def test_wait_that_runs_out_is_reported(n):
    """With a limit of 0 every wait of the products gives up at once: the blocks end by
    themselves, the inverse returns MSP_ERR_TIMEOUT, and the next one is right."""
    rp, ci, v = _system(n, 5)
    first = _inverse(rp, ci, v, 0, 0)
    _inverse(rp, ci, v, 0, 0, wait_ns=0, status=_native.MSP_ERR_TIMEOUT)
    torch.cuda.synchronize()
    assert torch.equal(_inverse(rp, ci, v, 0, 0), first)
