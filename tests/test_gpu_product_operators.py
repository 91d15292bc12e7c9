"""Products of several operators of one process, whose leaves differ in size (99-102, 189-192 and
303-306 rows): each keeps working after the others were used, in either order, for every
right-hand-side count of the kernels (the ones that several leaf sizes share take shared memory
by the leaf's rows).  Every repetition equals the operator's first product bit for bit (a product
adds in a fixed order), and that one agrees with the FP64-vector products within 1e-5 of the
absolute sums (the bar of the served paths' tests)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_operators_of_other_leaf_sizes_in_between(dtype, storage):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dt = torch.float32 if dtype == "f32" else torch.float64
    ops = []
    for grid, leaf in ((32, 110), (36, 64), (26, 64)):  # largest leaves first
        el = synth.disk_mesh(grid)
        H = hmat.HMatrix(hmat.ClusterTree(el, leaf, 2.0), el, 1.0, 0.25, 1e-6, storage)
        assert H.info()["u_entries"] > 0
        X = synth.rhs_normal(3 * el.N, 5 + leaf, 16).astype(np.float32)
        x = torch.from_numpy(X).cuda().to(dt)
        ref = torch.empty((16, 3 * el.N), dtype=torch.float64, device="cuda")
        H.matvec(x.double(), ref)
        A = np.abs(O.dense_matrix(el, 1.0, 0.25))
        ops.append((H, x, ref, np.linalg.norm(A @ np.abs(X).T.astype(np.float64), axis=0)))
    first = {}
    for order in ((0, 1, 2), (2, 1, 0), (0, 2, 1)):
        for nrhs in (16, 8, 4, 1, 3, 6, 11):
            for i in order:
                H, x, ref, scale = ops[i]
                y = torch.full((nrhs, x.shape[1]), float("nan"), dtype=dt, device="cuda")
                H.matvec(x[:nrhs].contiguous(), y)
                if (i, nrhs) in first:
                    assert torch.equal(y, first[i, nrhs]), (i, nrhs)
                first[i, nrhs] = y
                err = np.linalg.norm((y.double() - ref[:nrhs]).cpu().numpy(), axis=1) / scale[:nrhs]
                assert err.max() <= 1e-5, (i, nrhs, err)
    for H, *_ in ops:
        H.check()
