"""Face fluxes over the FP64 range: the flux of power-of-two scaled states is
the scaled flux (density s, pressure s c^2, velocity c, B c sqrt(s), psi c^2 sqrt(s)),
so the oracle at scale 1 is the reference everywhere.  The large scales leave
the exponent range of the fixed-point reciprocal and square root and take the
CUDA functions; supersonic and nearly still normal velocities take the outer
and the double-star branches.  Tolerance: 1e-12 relative L1 per component, as
every FP64 flux test."""
import numpy as np
import pytest

import oracle as orc
from paper_2510_24175_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s_exp,c_exp", [(0, 0), (-600, 0), (600, 0), (-966, 0), (966, 0),
                                         (0, -60), (0, 60)])
@pytest.mark.parametrize("normal", [1.0, 8.0, 0.01])
def test_flux_of_scaled_states(s_exp, c_exp, normal):
    import torch

    import paper_2510_24175_gb300 as m
    VL, VR = inputs.random_face_states(20_001, seed=77)
    d = 1
    VL[1 + d] *= normal
    VR[1 + d] *= normal
    ch, gamma = 1.7, 5.0 / 3.0
    ref = orc.interface_flux(VL, VR, d, ch, gamma)
    s, c, b = 2.0 ** s_exp, 2.0 ** c_exp, 2.0 ** (s_exp // 2 + c_exp)
    scale = np.array([s, c, c, c, b, b, b, s * c * c, b * c])[:, None]
    flux = np.array([s * c, s * c * c, s * c * c, s * c * c, b * c, b * c, b * c, s * c ** 3,
                     c * c * b])[:, None]
    tl, tr = (torch.from_numpy(V * scale).cuda() for V in (VL, VR))
    F = torch.empty_like(tl)
    m.mhd_flux_batch(tl, tr, F, d, ch * c, gamma)
    got = F.cpu().numpy() / flux
    err = np.abs(got - ref).sum(axis=1) / np.abs(ref).sum(axis=1)
    assert np.all(err <= 1e-12), err
