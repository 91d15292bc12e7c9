"""Products with a far field on leaves of every row-block count of the kernels: at most 102, 153,
192, 237 and 306 rows.  Every right-hand-side count of a kernel or a pass boundary, both storages:

* one FP64-vector product against the dense oracle: eps + 1e-6, with BF16 factors eps + 2^-8;
* FP64 vectors, several right-hand sides against their single products: both are compensated sums
  whose error is at most about (n u)^2 of the row's absolute sum, u = 2^-24, n < 100 terms an
  accumulator: 4e-11; 1e-11 of the absolute sums in the 2-norm is asked;
* FP32 vectors against the FP64-vector products of the same factors: 1e-5 of the absolute sums
  (FP32 accumulation, and 16 bits of the vectors on the tensor-core paths).

Then FP64 counts that leave a remainder on an operator whose coefficients are too many for padded
passes (two sets of passes), and on one where they are not, with the same bar."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu

E, NU = 1.0, 0.25


def need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("grid,leaf,rows", [(26, 64, 102), (32, 64, 153), (36, 64, 192), (40, 110, 237), (32, 110, 306)])
def test_leaf_sizes(grid, leaf, rows, storage):
    torch = need_gpu()
    el = synth.disk_mesh(grid)
    T = hmat.ClusterTree(el, leaf, 2.0)
    t = T.export()
    assert 3 * (t["end"] - t["begin"])[t["left"] < 0].max() == rows
    H = hmat.HMatrix(T, el, E, NU, 1e-6, storage)
    assert H.info()["u_entries"] > 0 and H.info()["v_entries"] > 0
    A = O.dense_matrix(el, E, NU)
    X = synth.rhs_normal(3 * el.N, 17 + rows, 19).astype(np.float32).astype(np.float64)
    x = torch.from_numpy(X).cuda()
    one = torch.empty_like(x)
    for k in range(19):
        y = torch.empty(3 * el.N, dtype=torch.float64, device="cuda")
        H.matvec(x[k].contiguous(), y)
        one[k] = y
    ref = X @ A.T
    err = np.linalg.norm(one.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 1e-6 + (1e-6 if storage == "f32" else 2.0 ** -8), err
    scale = np.linalg.norm(np.abs(A) @ np.abs(X).T, axis=0)
    for dt, bar in ((torch.float64, 1e-11), (torch.float32, 1e-5)):
        for nrhs in (1, 2, 3, 4, 5, 6, 8, 9, 11, 13, 16, 17, 19):
            y = torch.full((nrhs, 3 * el.N), float("nan"), dtype=dt, device="cuda")
            H.matvec(x[:nrhs].to(dt).contiguous(), y)
            err = np.linalg.norm((y.double() - one[:nrhs]).cpu().numpy(), axis=1) / scale[:nrhs]
            assert err.max() <= bar, (dt, nrhs, err)
    H.check()


@pytest.mark.parametrize("grid", [48, 96])
def test_f64_remainders(grid):
    torch = need_gpu()
    el = synth.disk_mesh(grid)
    H = hmat.HMatrix(hmat.ClusterTree(el, 64, 2.0), el, E, NU, 1e-6, "f32")
    i = H.info()
    assert (i["near_entries"] + i["u_entries"] + i["v_entries"] > 2 ** 24) == (grid == 96)
    X = synth.rhs_normal(3 * el.N, 23, 31)
    x = torch.from_numpy(X).cuda()
    one = torch.empty_like(x)
    for k in range(31):
        y = torch.empty(3 * el.N, dtype=torch.float64, device="cuda")
        H.matvec(x[k].contiguous(), y)
        one[k] = y
    for nrhs in (5, 7, 10, 14, 15, 21, 31):
        for rep in range(3):  # the split leaves' arrival counts are left clean
            y = torch.full((nrhs, 3 * el.N), float("nan"), dtype=torch.float64, device="cuda")
            H.matvec(x[:nrhs].contiguous(), y)
            err = (y - one[:nrhs]).norm(dim=1) / one[:nrhs].norm(dim=1)
            assert err.max().item() <= 1e-11, (nrhs, rep, err)
    H.check()
