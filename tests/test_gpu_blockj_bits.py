"""Block-Jacobi inverses entry by entry: Gauss-Jordan in FP32 with partial pivoting over the rows
not yet used (ties: the lowest), each entry by fused multiply-adds in the order of the columns, on
the stored blocks.  A CPU run of that recurrence (numpy, the fused operation as an exact product,
a sum rounded to odd in FP64 and one rounding to FP32: Boldo and Melquiond, 2008) must give the
kernel's inverse bit for bit, whatever panels it works in: leaves of 18 to 192 rows, full and
partial panels.  And a block that becomes singular at its last columns is refused."""
import numpy as np
import pytest

from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


def need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def fma32(a, b, c):
    p = a.astype(np.float64) * b.astype(np.float64)
    c = c.astype(np.float64)
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)
    even = (np.ascontiguousarray(s).view(np.int64) & 1) == 0
    s = np.where((e != 0) & even, np.nextafter(s, np.where(e > 0, np.inf, -np.inf)), s)
    return s.astype(np.float32)


def gauss_jordan(a):
    n = a.shape[0]
    a = a.copy()
    free = np.ones(n, bool)
    p = np.empty(n, int)
    for k in range(n):
        c = a[:, k].copy()
        p[k] = np.argmax(np.where(free, np.abs(c), -1.0))
        free[p[k]] = False
        inv = np.float32(1.0) / c[p[k]]
        r = a[p[k]] * inv
        r[k] = inv
        a = fma32(-c[:, None], r[None, :], a)
        a[:, k] -= c
        a[p[k]] = r
    x = np.empty_like(a)
    x[:, p] = a[p]  # unknown k: row p_k; its coefficient of equation p_q: column q
    return x


def leaf_rows(T):
    t = T.export()
    return [(3 * t["perm"][t["begin"][q]:t["end"][q], None] + np.arange(3)).ravel() for q in np.flatnonzero(t["left"] < 0)]


def stored_blocks(torch, H, rows, ndof):
    """The FP32 entries of every diagonal block, by products with unit vectors (exact in FP64)."""
    blocks = [np.empty((len(r), len(r)), np.float32) for r in rows]
    for j0 in range(0, max(map(len, rows)), 16):
        x = torch.zeros((16, ndof), dtype=torch.float64, device="cuda")
        y = torch.empty_like(x)
        for q, r in enumerate(rows):  # one leaf at a time: its columns only
            x.zero_()
            cols = range(j0, min(j0 + 16, len(r)))
            for k, j in enumerate(cols):
                x[k, r[j]] = 1.0
            if len(cols):
                H.matvec(x, y)
                blocks[q][:, j0:j0 + len(cols)] = y[:len(cols)].cpu().numpy()[:, r].T
    return blocks


@pytest.mark.parametrize("grid,leaf", [(8, 8), (10, 16), (12, 30), (20, 42), (32, 64), (36, 64)])
def test_inverse_bits(grid, leaf):
    torch = need_gpu()
    el = synth.disk_mesh(grid)
    T = hmat.ClusterTree(el, leaf, 2.0)
    H = hmat.HMatrix(T, el, 1.0, 0.25, 1e-6, "f32")
    n = 3 * el.N
    rows = leaf_rows(T)[:6]
    rng = np.random.default_rng(70 + leaf)
    k = synth.k_loguniform(el.N, 71, 1.0, 2.0 / grid)
    cep = rng.normal(size=(el.N, 3, 3))
    cep[:, np.arange(3), np.arange(3)] = 0.0
    kd, cd = torch.from_numpy(k).cuda(), torch.from_numpy(cep).cuda()
    # (C^ep without a diagonal: the library adds that to k in FP64)
    blocks = stored_blocks(torch, H, rows, n)
    inv = []
    for r, b in zip(rows, blocks):
        e = r // 3
        b[np.arange(len(r)), np.arange(len(r))] -= k[e].astype(np.float32)
        for u in np.unique(e):
            i = np.flatnonzero(e == u)
            b[np.ix_(i, i)] -= cep[u].astype(np.float32)
        inv.append(gauss_jordan(b))
    top = max(map(len, rows))
    for m0 in range(0, top, 16):
        x = np.zeros((16, n))
        for r in rows:
            for q, m in enumerate(range(m0, min(m0 + 16, len(r)))):
                x[q, r[m]] = 1.0
        z = torch.empty((16, n), dtype=torch.float64, device="cuda")
        H.precond_apply(torch.from_numpy(x).cuda(), z, k=kd, cep=cd)
        z = z.cpu().numpy()
        for r, a in zip(rows, inv):
            cols = min(16, len(r) - m0)
            if cols > 0:
                assert np.array_equal(z[:cols, r].T, a[:, m0:m0 + cols].astype(np.float64)), (len(r), m0)


@pytest.mark.parametrize("grid,leaf", [(8, 16), (12, 32), (16, 64)])
def test_a_block_singular_past_its_first_panel_is_refused(grid, leaf):
    """Every element of a leaf but the last gets a stiffness of 2^100 and E is tiny, so the last
    element's 3x3 block stays what it is through the earlier columns (what they subtract
    underflows): zero, its own C^ep being its stored self block."""
    torch = need_gpu()
    el = synth.disk_mesh(grid)
    T = hmat.ClusterTree(el, leaf, 2.0)
    H = hmat.HMatrix(T, el, 2.0 ** -30, 0.25, 1e-6, "f32")
    n = 3 * el.N
    rows = leaf_rows(T)
    last = rows[0][-3:]
    assert len(rows[0]) > 16
    k = np.full(el.N, 2.0 ** 100)
    k[last[0] // 3] = 0.0
    x = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    x[np.arange(3), last] = 1.0
    H.matvec(x, y)
    cep = np.zeros((el.N, 3, 3))
    cep[last[0] // 3] = y.cpu().numpy()[:, last].T
    r = torch.ones(n, dtype=torch.float64, device="cuda")
    out = torch.empty_like(r)
    kd = torch.from_numpy(k).cuda()
    with pytest.raises(hmat.HMError) as ei:
        H.precond_apply(r, out, k=kd, cep=torch.from_numpy(cep).cuda())
    assert ei.value.status == hmat.HM_EBREAKDOWN
    cep[last[0] // 3, 0, 0] -= 1.0  # not singular any more in that column, still in the others
    cep[last[0] // 3, 1, 1] -= 1.0
    cep[last[0] // 3, 2, 2] -= 1.0
    H.precond_apply(r, out, k=kd, cep=torch.from_numpy(cep).cuda())
    assert torch.isfinite(out).all()
