"""Face fluxes between a light hot side and a dense cold one, pressures of order 1 and
density ratios up to 10^8, either side dense, subsonic normal speeds on each side's
own scale, without field and with one of order 1, against the FP64 oracle.  Error
bound: 450 units in the last place (2^-53, 2^-24) of the face's flux scale, about
150 roundings of up to three scales each; scales: the larger density, energy and
speed of the two sides and their products, S - S_M being of the order of the speed
(no cancellation is inherent in these states).  The FP64 bound allows for the
oracle's own rounding as well: it adds up wave jumps S (U* - U), in the momenta
terms of the dense side's momentum times the light side's speed."""
import numpy as np
import pytest

import oracle as orc

pytestmark = pytest.mark.gpu

N = 200_000


def faces(field, dense_right, seed):
    rng = np.random.default_rng(seed)
    V = np.zeros((2, 9, N))
    V[0, 0] = 10.0 ** rng.uniform(-8, 0, N)
    V[1, 0] = 1.0
    V[:, 7] = np.exp(rng.uniform(-1, 1, (2, N)))
    c = np.sqrt(V[:, 7] / V[:, 0])
    V[:, 1:4] = 0.3 * rng.normal(size=(2, 3, N)) * c[:, None]
    V[:, 4:7] = field * rng.normal(size=(2, 3, N))
    V[:, 8] = 0.01 * field * rng.normal(size=(2, N))
    return V if dense_right else V[::-1].copy()


def scales(V, gamma, ch):
    rho, B2 = V[:, 0], (V[:, 4:7] ** 2).sum(axis=1)
    v2 = (V[:, 1:4] ** 2).sum(axis=1)
    c = (np.sqrt((gamma * V[:, 7] + B2) / rho) + np.sqrt(v2)).max(axis=0)
    E = (V[:, 7] * gamma / (gamma - 1) + 0.5 * rho * v2 + B2).max(axis=0)
    r, B = rho.max(axis=0), np.sqrt(E) * c + ch * np.sqrt(E)
    jump = r * c * np.sqrt(np.take_along_axis(v2, rho.argmax(axis=0)[None], axis=0)[0])
    base = np.stack([r * c, E, E, E, B, B, B, E * c, ch * ch * np.sqrt(E)])
    return base, np.stack([0 * E, jump, jump, jump] + [0 * E] * 5)


@pytest.mark.parametrize("field", [0.0, 1.0])
@pytest.mark.parametrize("dense_right", [False, True])
@pytest.mark.parametrize("direction", [0, 1, 2])
def test_flux_across_a_density_contrast(field, dense_right, direction):
    import torch
    import paper_2510_24175_gb300 as m
    gamma, ch = 5.0 / 3.0, 1.7
    V = faces(field, dense_right, seed=21)
    for dtype, ulp in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
        L, R = (torch.from_numpy(v).to(dtype).cuda().contiguous() for v in V)
        F = torch.empty_like(L)
        m.mhd_flux_batch(L, R, F, direction, ch, gamma)
        W = np.stack([L.double().cpu().numpy(), R.double().cpu().numpy()])
        ref = orc.interface_flux(W[0], W[1], direction, ch, gamma)
        base, oracle_jumps = scales(W, gamma, ch)
        if dtype == torch.float64:
            base += oracle_jumps
        err = np.abs(F.double().cpu().numpy() - ref) / base
        assert np.isfinite(err).all() and err.max() <= 450 * ulp, (dtype, err.max(axis=1) / ulp)
