"""The interface update where its outputs are known to the last bits.

* Perfect plasticity: an apex or tensile return holds the normal traction (c / f or sigma_t), so
  dT'_n / d(Delta delta_n) = K_n - K_n (f K_n / (f K_n)) is exactly zero for any K_n and f.
* chi_s and chi_t where they grow are the magnitudes of the delta^p that the step returns."""
import numpy as np
import pytest

from oracle import interface as I
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


def update(kw, states):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = hmat.interface_update(kw, *[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in states], counts=True)
    return [a.cpu().numpy() for a in out[:5]] + [out[5]]


@pytest.mark.parametrize("sigp", [0.25, 1.0])
def test_held_normal_traction_has_no_stiffness(sigp):
    rng = np.random.default_rng(5)
    seen = 0
    for q in range(32):
        f = rng.uniform(0.2, 0.9)
        kw = dict(Ks=rng.uniform(5, 20), Kn=rng.uniform(5, 40), fp=f, fr=f, psip=0.1, dc=1e300, cp=0.2, sigp=sigp,
                  wc=1e300, alphaR=0.0)
        T1, dp1, chi1, cep, mode, cnt = update(kw, synth.interface_states(1024, 90 + q))
        held = (mode == I.APEX) | (mode == I.TENSILE)
        seen += held.sum()
        assert (cep[held, 2, 2] == 0.0).all(), (q, np.abs(cep[held, 2, 2]).max())
    assert seen > 1000


@pytest.mark.parametrize("name", list(synth.INTERFACE_PARAMS))
def test_grown_internal_variables_are_rounded_square_roots(name):
    """chi_s and chi_t where a return made them grow: the magnitudes of delta^p, each the rounded
    square root of a sum of squares whose roundings count half.  Independent roundings of 0.41 u rms
    (u = 2^-53, mantissas spread over a binade) make 0.41 (1 + 3/4)^1/2 = 0.54 u rms for three
    squares at most; 0.58 u is asked of every mode with 1,000 such points."""
    states = synth.interface_states(100000, 3)
    T1, dp1, chi1, cep, mode, cnt = update(synth.INTERFACE_PARAMS[name], states)
    dp = dp1.astype(np.longdouble)
    tested = 0
    for kind in (I.COULOMB, I.TENSILE, I.APEX):
        for c, n in ((0, 2), (1, 3)):
            ref = np.sqrt((dp[:, :n] ** 2).sum(axis=1))
            grown = (mode == kind) & (chi1[:, c] > states[2][:, c])
            if grown.sum() < 1000:
                continue
            err = ((chi1[grown, c] - ref[grown]) / ref[grown] * 2.0 ** 53).astype(np.float64)
            assert np.sqrt((err ** 2).mean()) <= 0.58, (kind, c, np.sqrt((err ** 2).mean()))
            tested += 1
    assert tested >= 2


@pytest.mark.parametrize("Ks", [7.0, 10.0, 1.0 / 3.0, 13.7])
@pytest.mark.parametrize("fp", [0.0, 0.4])
def test_frictionless_contact_slips(Ks, fp):
    """A pre-existing fracture without friction (or softened to none by the step's slip) under
    compression: g is zero where the shear traction vanishes, and the return is the Coulomb one
    with all of the trial shear inelastic, never an open state.  Bars: a few roundings of the
    trial and shear tractions, of the slip and of K_s."""
    rng = np.random.default_rng(int(100 * Ks) + int(10 * fp))
    n = 20000
    kw = dict(Ks=Ks, Kn=2 * Ks, fp=fp, fr=0.0, psip=0.0, dc=1e-6 if fp else 0.2, cp=0.0, sigp=0.0, wc=0.0, alphaR=0.0)
    T = np.c_[rng.normal(size=(n, 2)) * 0.2, -rng.uniform(0.5, 1.5, n)]
    dp, chi = np.zeros((n, 3)), np.zeros((n, 3))
    dd = np.c_[rng.normal(size=(n, 2)) * 0.08, rng.normal(size=n) * 1e-3]
    tr = T + np.array([Ks, Ks, 2 * Ks]) * dd
    tau = np.hypot(tr[:, 0], tr[:, 1])
    assert (tr[:, 2] < 0).all() and (tau > 1.1 * fp * np.abs(tr[:, 2])).sum() > 1000
    T1, dp1, chi1, cep, mode, cnt = update(kw, (T, dp, chi, dd))
    slips = tau > 1.1 * fp * np.abs(tr[:, 2]) + 2 * Ks * kw["dc"] * (fp > 0)
    u = 2.0 ** -53
    assert (mode[slips] == I.COULOMB).all() and cnt[3] == cnt[4] == cnt[5] == 0
    assert (np.abs(T1[slips, :2]).max(axis=1) <= 16 * u * tau[slips]).all()
    assert np.abs(T1[slips, 2] - tr[slips, 2]).max() <= 8 * u * 2
    trial = 4 * u * (np.abs(T) + Ks * np.abs(dd))[:, :2].max(axis=1)  # the trial traction's own roundings
    assert (np.abs(dp1[slips, :2] - tr[slips, :2] / Ks).max(axis=1) <= (16 * u * tau + trial)[slips] / Ks).all()
    assert np.abs(cep[slips][:, :2, :2]).max() <= 64 * u * Ks and np.abs(cep[slips, 2, 2] - 2 * Ks).max() <= 8 * u * 2 * Ks
    P = I.Params(**kw)
    q = np.flatnonzero(slips)[:150]
    assert np.array_equal(mode[q], [I.update(P, T[e], dp[e], chi[e], dd[e])["mode"] for e in q])
