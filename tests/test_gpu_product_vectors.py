"""BF16 factors with 2 to 15 FP32 right-hand sides (and the last pass of 27): the vectors are
used as they are.  Every right-hand side is c times a unit vector, c = 1 + 2^-9 + 2^-17 - 2^-23,
whose split into two BF16 numbers would lose 2^-17 of it, so the far rows of its product are one
product per rank entry and a sum of `rank` terms: each row within (rank + 3) 2^-24 of
sum_l |U_l| |V_l| c (a rounding of V c, one of each product and sum; 1 % for the factors' BF16
rounding) of the FP64-vector product of the same stored factors.  Leaves of 120, 192 and 237 rows:
one size for each variant of the kernels."""
import numpy as np
import pytest

from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,leaf", [(40, 64), (36, 64), (40, 110)])
@pytest.mark.parametrize("nrhs", [2, 7, 9, 12, 15, 27])
def test_vectors_keep_fp32(grid, leaf, nrhs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(grid)
    T = hmat.ClusterTree(el, leaf, 2.0)
    H = hmat.HMatrix(T, el, 1.0, 0.25, 1e-6, "bf16")
    t = T.export()
    dof = np.random.default_rng(8 + nrhs).choice(3 * el.N, nrhs, replace=False)
    c = 1 + 2.0 ** -9 + 2.0 ** -17 - 2.0 ** -23
    X = np.zeros((nrhs, 3 * el.N))
    X[np.arange(nrhs), dof] = c
    bar = np.full((nrhs, 3 * el.N), np.inf)
    rows = lambda q: (3 * t["perm"][t["begin"][q]:t["end"][q], None] + np.arange(3)).ravel()
    for b, (s, q) in enumerate(t["far"]):
        uv = H.far_factor_arrays(b, t["end"][s] - t["begin"][s], t["end"][q] - t["begin"][q])
        if uv is None:
            continue
        i, j = rows(s), rows(q)
        for k in np.flatnonzero(np.isin(dof, j)):
            v = np.abs(uv[1][np.flatnonzero(j == dof[k])[0]]) * c
            bar[k, i] = 1.01 * (uv[0].shape[1] + 3) * 2.0 ** -24 * (np.abs(uv[0]) @ v)
    far = np.isfinite(bar)
    assert far.mean() > 0.3
    far[:nrhs // 16 * 16] = False  # full passes of 16 take the tensor cores
    y = []
    for dt in (torch.float64, torch.float32):
        x = torch.from_numpy(X).cuda().to(dt)
        out = torch.empty_like(x)
        H.matvec(x, out)
        y.append(out.double().cpu().numpy())
    err = np.abs(y[1] - y[0])
    assert (err[far] <= bar[far]).all()
