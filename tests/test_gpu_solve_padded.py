"""Mixed solves of right-hand-side counts that the FP32 products pad (2, 3, 5, 11), back to back on
one operator with vectors that converge at different iterations, so that the last products of a
cycle are skipped while the next solve's kernels are already queued: every repetition equals the
first bit for bit (the kernels add in a fixed order), every residual is within the tolerance, with
and without a far field."""
import pytest

from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eta", [2.0, 1e-3])
@pytest.mark.parametrize("nrhs", [2, 3, 5, 11])
def test_padded_solves_repeat(nrhs, eta):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(24)
    H = hmat.HMatrix(hmat.ClusterTree(el, 32, eta), el, 1.0, 0.25, 1e-6, "both")
    k = torch.from_numpy(synth.k_loguniform(el.N, 91, 1.0, 1.0 / 12)).cuda()
    g = torch.Generator(device="cuda").manual_seed(92)
    b = torch.randn((2, nrhs, 3 * el.N), generator=g, device="cuda", dtype=torch.float64)
    b[:, 0] = torch.ones(3 * el.N, device="cuda", dtype=torch.float64)  # a smooth one converges first
    first = [None, None]
    for rep in range(10):
        for q in range(2):
            x = torch.empty_like(b[q])
            H.solve(b[q], x, k=k, tol=1e-8, precond="blockj", mode="mixed")
            if first[q] is None:
                first[q] = x
                y = torch.empty_like(x)
                H.matvec(x, y)
                res = (y - k.repeat_interleave(3) * x - b[q]).norm(dim=1) / b[q].norm(dim=1)
                assert res.max().item() <= 2e-8, res
            assert torch.equal(x, first[q]), (rep, q)
