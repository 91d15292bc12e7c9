"""The interface update where its outputs are known to the last bits.

* Perfect plasticity: an apex or tensile return holds the normal traction (c / f or sigma_t), so
  dT'_n / d(Delta delta_n) = K_n - K_n (f K_n / (f K_n)) is exactly zero for any K_n and f."""
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
