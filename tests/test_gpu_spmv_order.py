"""msp_spmv works on the caller's vectors directly where it may (x on a 16-byte boundary, not
overlapping y) and through colour-ordered copies elsewhere: both give the same bits, for every
block size, with and without long well rows, and with y = x."""
import numpy as np
import pytest

from synthetic import box_jacobian

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_08594_gb300 as msp  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("wells", [0, 2])
@pytest.mark.parametrize("b", [1, 2, 3, 4, 5, 6, 7, 8])
def test_aligned_shifted_and_overlapping_vectors_agree(b, wells):
    a = box_jacobian(5, 4, 19, b, 40 + b, layered=True, kz_ratio=0.1, n_wells=wells)
    s = msp.Solver(a.nb, b, *(torch.from_numpy(x).to(DEV) for x in
                              (a.row_ptr, a.col_idx, a.values.reshape(-1))), coarse_max=50)
    x = np.random.default_rng(b).normal(size=a.n)
    buf = torch.zeros(2 * a.n + 16, dtype=torch.float64, device=DEV)
    out = []
    for off in (0, 1):  # 16-byte boundary, or 8 bytes past one
        buf[off:off + a.n] = torch.from_numpy(x).to(DEV)
        y = torch.full((a.n,), float("nan"), dtype=torch.float64, device=DEV)
        s.spmv(buf[off:off + a.n], y)
        out.append(y.cpu().numpy())
    inplace = torch.from_numpy(x).to(DEV)
    s.spmv(inplace, inplace)
    out.append(inplace.cpu().numpy())
    buf[:a.n] = torch.from_numpy(x).to(DEV)  # y starts inside x
    s.spmv(buf[:a.n], buf[a.n // 2:a.n // 2 + a.n])
    out.append(buf[a.n // 2:a.n // 2 + a.n].cpu().numpy())
    for y in out[1:]:
        assert np.array_equal(y, out[0])
    # one rounding per product and sum: n terms of a row, each within 2^-53 of |A| |x|
    ref = a.to_scipy() @ x
    terms = int(np.diff(a.row_ptr).max()) * b
    bound = 2 * terms * 2.0 ** -53 * (abs(a.to_scipy()) @ np.abs(x))
    assert (np.abs(out[0] - ref) <= bound).all()
    s.close()
