"""Block-Jacobi inverses on every register tile of the builder (leaves of 3 to 192 rows, full
and partial panels of eight columns), through hm_precond_apply, with k and with C^ep.

Reference: numpy's FP64 solve of every leaf block of the oracle's dense tangent.  Bar per leaf:
4 n cond(B) 2^-24 of the leaf's solution (Gauss-Jordan with partial pivoting in FP32 on n rows,
the blocks rounded to FP32, an FP32 product).  A block of zeros is still refused."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu

E, NU = 1.0, 0.25


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("with_cep", [False, True])
@pytest.mark.parametrize("leaf", [1, 2, 3, 10, 11, 13, 21, 22, 32, 43, 53, 54, 64])
def test_leaf_inverses(leaf, with_cep):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(18)
    T = hmat.ClusterTree(el, leaf, 2.0)
    H = hmat.HMatrix(T, el, E, NU, 1e-6, "f32")
    A = O.dense_matrix(el, E, NU)
    rng = np.random.default_rng(60 + leaf)
    k = synth.k_loguniform(el.N, 61, E, 1.0 / 9)
    cep = rng.normal(size=(el.N, 3, 3)) * 2.0 if with_cep else None
    r = rng.normal(size=3 * el.N)
    z = torch.empty(3 * el.N, dtype=torch.float64, device="cuda")
    H.precond_apply(dev(r), z, k=dev(k), cep=dev(cep) if with_cep else None)
    z = z.cpu().numpy()
    B = A - np.diag(np.repeat(k, 3))
    if with_cep:
        for e in range(el.N):
            B[3 * e:3 * e + 3, 3 * e:3 * e + 3] -= cep[e]
    t = T.export()
    for q in np.flatnonzero(t["left"] < 0):
        i = O.dof_index(t["perm"][t["begin"][q]:t["end"][q]])
        b = B[np.ix_(i, i)]
        ref = np.linalg.solve(b, r[i])
        bar = 4 * len(i) * np.linalg.cond(b) * 2.0 ** -24
        err = np.linalg.norm(z[i] - ref) / np.linalg.norm(ref)
        assert err <= bar, (leaf, q, err, bar)


def test_zero_block_is_refused():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    el = synth.disk_mesh(6)
    H = hmat.HMatrix(hmat.ClusterTree(el, 1, 2.0), el, E, NU, 1e-6, "f32")
    A = O.dense_matrix(el, E, NU)
    cep = np.zeros((el.N, 3, 3))
    cep[5] = A[15:18, 15:18].astype(np.float32)  # the stored self block of element 5: nothing is left of it
    r = torch.ones(3 * el.N, dtype=torch.float64, device="cuda")
    own = torch.from_numpy(cep).cuda()
    out = torch.empty_like(r)
    # the library's self block may differ from the oracle's by an FP32 ulp: read it back by a unit product
    for m in range(3):
        e = torch.zeros_like(r)
        e[15 + m] = 1.0
        H.matvec(e, out)
        own[5, :, m] = out[15:18]
    with pytest.raises(hmat.HMError) as ei:
        H.precond_apply(r, out, cep=own)
    assert ei.value.status == hmat.HM_EBREAKDOWN
