"""The interface update in other units: tractions times 2^30 and displacements times 2^-20 (SI
sizes of a rock joint) and 2^-80 (whose squares FP32 cannot hold, so that the FP32 guess of the
multiplier is worthless and the FP64 iteration starts from anywhere).  Powers of two scale every
FP64 quantity of the law exactly, so the oracle's unscaled step, scaled, is the reference: modes
bit for bit, state to 1e-12 of the traction and DD scales, C^ep to 1e-9 of the stiffness (the
bars of the unscaled test).  Two inconsistent states are among them (chi below |delta^p|)."""
import numpy as np
import pytest

from oracle import interface as I
from paper_2605_14397_gb300 import hmat, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", list(synth.INTERFACE_PARAMS))
@pytest.mark.parametrize("pa,pd", [(30, -20), (0, -80)])
def test_scaled_units(name, pa, pd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, d = 2.0 ** pa, 2.0 ** pd
    kw = synth.INTERFACE_PARAMS[name]
    T, dp, chi, dd = synth.interface_states(257, 47)
    chi[:40, :2] *= 0.5
    rT, rdp, rchi, rmode, rcep = I.step_all(I.Params(**kw), T, dp, chi, dd)
    up = dict(kw, Ks=kw["Ks"] * a / d, Kn=kw["Kn"] * a / d, cp=kw["cp"] * a, sigp=kw["sigp"] * a,
              dc=kw["dc"] if kw["dc"] > 1e100 else kw["dc"] * d, wc=kw["wc"] if kw["wc"] > 1e100 else kw["wc"] * d)
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (T * a, dp * d, chi * d, dd * d)]
    T1, dp1, chi1, cep, mode, cnt = hmat.interface_update(up, *dev, counts=True)
    assert cnt[5] == 0
    assert np.array_equal(mode.cpu().numpy(), rmode)
    assert np.abs(T1.cpu().numpy() / a - rT).max() <= 1e-12 * max(1.0, np.abs(rT).max())
    assert np.abs(dp1.cpu().numpy() / d - rdp).max() <= 1e-12 * max(0.1, np.abs(rdp).max())
    assert np.abs(chi1.cpu().numpy() / d - rchi).max() <= 1e-12 * max(0.1, np.abs(rchi).max())
    assert np.abs(cep.cpu().numpy() * (d / a) - rcep).max() <= 1e-9 * max(kw["Ks"], kw["Kn"])
