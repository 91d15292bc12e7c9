"""FP64-vector products of 1 to 16 right-hand sides: every pass width (1 to 4, and counts cut
into several passes) on leaves of every row-block count of the kernels (fewer than 64 rows
to more than 192) and both factor precisions.

Every right-hand side of a product must match its own single-RHS product, which the stored
operator checks entry by entry elsewhere.  Bar: both are compensated sums whose error is at
most about (n u)^2 of the row's absolute sum, u = 2^-24, n the terms one accumulator adds
(at most 948 columns over 14 warps and their partial sums: n < 100): 4e-11; 1e-11 of the
absolute sums in the 2-norm is asked.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu

E, NU = 1.0, 0.25


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("leaf", [8, 21, 43, 64, 110])
def test_f64_passes_match_single_rhs(leaf, storage):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(20)  # 316 elements: leaves of 5 to 79 elements
    T = hmat.ClusterTree(el, leaf, 1.0)
    H = hmat.HMatrix(T, el, E, NU, 1e-6, storage)
    A = np.abs(O.dense_matrix(el, E, NU))
    X = synth.rhs_normal(3 * el.N, 31 + leaf, 16)
    x = torch.from_numpy(X).cuda()
    one = torch.empty_like(x)
    for k in range(16):
        xk, yk = x[k].contiguous(), torch.empty(3 * el.N, dtype=torch.float64, device="cuda")
        H.matvec(xk, yk)
        one[k] = yk
    scale = np.linalg.norm(A @ np.abs(X).T, axis=0)
    for nrhs in (2, 3, 4, 5, 7, 16):
        y = torch.empty((nrhs, 3 * el.N), dtype=torch.float64, device="cuda")
        H.matvec(x[:nrhs].contiguous(), y)
        err = np.linalg.norm((y - one[:nrhs]).cpu().numpy(), axis=1) / scale[:nrhs]
        assert err.max() <= 1e-11, (nrhs, err)
    H.check()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("leaf", [8, 33, 42, 64, 110])
def test_f32_counts_match_f64_vectors(leaf, storage):
    """FP32 vectors, every count a pass is padded from (2 .. 16) and counts cut into several
    passes, against the FP64-vector product of the same stored factors: every right-hand side
    within 1e-5 of its absolute sums (FP32 accumulation, and 16 bits of the vectors on the
    tensor-core paths: the bar of the served paths' tests)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(26)
    T = hmat.ClusterTree(el, leaf, 1.0)
    H = hmat.HMatrix(T, el, E, NU, 1e-6, storage)
    A = np.abs(O.dense_matrix(el, E, NU))
    X = synth.rhs_normal(3 * el.N, 71 + leaf, 19).astype(np.float32)
    x = torch.from_numpy(X).cuda()
    ref = torch.empty((19, 3 * el.N), dtype=torch.float64, device="cuda")
    H.matvec(x.double(), ref)
    scale = np.linalg.norm(A @ np.abs(X).T.astype(np.float64), axis=0)
    for nrhs in (1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 19):
        y = torch.full((nrhs, 3 * el.N), float("nan"), dtype=torch.float32, device="cuda")
        H.matvec(x[:nrhs].contiguous(), y)
        err = np.linalg.norm((y.double() - ref[:nrhs]).cpu().numpy(), axis=1) / scale[:nrhs]
        assert err.max() <= 1e-5, (nrhs, err)
    H.check()


def test_near_field_only_products_follow_their_operand():
    """An operator without admissible blocks: phase 2 comes straight after the kernel that writes
    its operand.  500 products of changing vectors, each within (eps + 1e-6) of the oracle's."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(24)
    H = hmat.HMatrix(hmat.ClusterTree(el, 64, 1e-3), el, E, NU, 1e-6, "f32")
    assert H.info()["u_entries"] == 0
    A = torch.from_numpy(O.dense_matrix(el, E, NU)).cuda()
    g = torch.Generator(device="cuda").manual_seed(9)
    for dt, nrhs in ((torch.float32, 1), (torch.float64, 1), (torch.float32, 3)):
        xs = torch.randn((500, nrhs, 3 * el.N), generator=g, device="cuda", dtype=dt)
        ys = torch.empty_like(xs)
        for q in range(500):
            H.matvec(xs[q], ys[q])
        ref = xs.double() @ A.T
        err = (ys.double() - ref).norm(dim=2) / ref.norm(dim=2)
        assert err.max().item() <= 2e-6, (dt, nrhs, err.max().item())
