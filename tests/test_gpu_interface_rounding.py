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
