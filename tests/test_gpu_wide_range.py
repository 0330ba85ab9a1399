"""FP32 contexts over wide ranges of the incident field, against a PRD_FP64 context of the same
problem: what FP32 tiles and FP32-level products promise at any exponent, not only beside a row's
or a direction's largest value.

The redistribution is coherent in the wings, so a field that spans 2^40 over frequency leaves an
emissivity that spans as much, frequency by frequency made of the field near it.  Without
elastic collisions (no R_III, which spreads the core over the wings) every element is compared
with its own size: perturbing the field by 1e-7 moves the elements by at most 1e-6 (evaluated
with the oracle), FP32 tiles, field and frame changes are some ten such roundings and at most 240
partial sums of 2^-23 a product chain; 1e-4 covers their product.  (Operands under one scale a row,
which hold a value to 2^-38 of the row's largest, exceed it.)"""
import numpy as np
import pytest
import torch

from paper_2505_20968_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cfg(nnu, mode=inputs.MODE_AD, n_z=2, n_mu=1, n_chi=3, coherent=True):
    cfg = inputs.hi_lya(n_z=n_z, n_core=nnu - 6, n_wing=6, n_mu_half=n_mu, n_chi=n_chi, seed=41, mode=mode)
    return dict(cfg, atm=dict(cfg["atm"], r_el=np.zeros(n_z))) if coherent else cfg


@pytest.mark.parametrize("nnu", [40, 100, 150, 200])
@pytest.mark.parametrize("tensor_cores", [True, False])
@pytest.mark.parametrize("sign", [1, -1])
def test_field_spanning_2_40_over_frequency(nnu, tensor_cores, sign):
    from paper_2505_20968_gb300.binding import PRD
    P, D = PRD(_cfg(nnu), precision="fp32", device=0), PRD(_cfg(nnu), precision="fp64", device=0)
    P.set_tensor_cores(tensor_cores)
    x = torch.zeros(P.shape, dtype=torch.float64, device="cuda")
    e = sign * 40.0 * (torch.arange(nnu, device="cuda", dtype=torch.float64) / (nnu - 1) - 0.5)
    x[..., 0] = torch.exp2(e)
    x = x.float().double()
    out = P.apply_sigma(x.float())[..., 0].double()
    ref = D.apply_sigma(x)[..., 0]
    P.device_status()
    # the intensity that the field near a frequency gives (tails where the tiles oscillate about zero are
    # compared with a thousandth of the field)
    size = torch.maximum(ref.abs(), 1e-3 * x[..., 0])
    assert float(((out - ref).abs() / size).max()) < 1e-4
    P.close()
    D.close()


@pytest.mark.parametrize("nnu,n_mu,n_chi,mode", [
    (9, 1, 3, inputs.MODE_AD), (33, 2, 4, inputs.MODE_AD), (65, 2, 3, inputs.MODE_AD), (128, 1, 4, inputs.MODE_AD),
    (129, 1, 4, inputs.MODE_AD), (161, 1, 4, inputs.MODE_AD), (193, 1, 3, inputs.MODE_AD), (224, 1, 3, inputs.MODE_AD),
    (21, 4, 8, inputs.MODE_AA), (150, 2, 4, inputs.MODE_AA)])
def test_fp32_contraction_at_tile_edges_matches_fp64(nnu, n_mu, n_chi, mode):
    """Row counts at the edges of the tiles, of the rows beyond 128 and of their packing; the
    bound of the FP32 CUDA-core contraction, 1e-6 of each height's largest emissivity."""
    from paper_2505_20968_gb300.binding import PRD
    cfg = _cfg(nnu, mode, 2, n_mu, n_chi, coherent=False)
    P, D = PRD(cfg, precision="fp32", device=0), PRD(cfg, precision="fp64", device=0)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 6, 0.1, 1.0)).to("cuda", torch.float32)
    x[:, -1, :, 1] = 0.0
    out, ref = P.apply_sigma(x).double(), D.apply_sigma(x.double())
    P.device_status()
    for z in range(P.nz):
        assert float((out[z] - ref[z]).abs().max() / ref[z, ..., 0].abs().max()) < 1e-6, z
    P.close()
    D.close()


@pytest.mark.parametrize("nnu", [27, 150])
def test_one_direction_and_stokes_parameter_at_any_scale(nnu):
    """The field in one direction and Stokes parameter alone, times a power of two: the emissivity
    scales along (products, sums and roundings do; R_III's FP64 sums may be taken in another order)."""
    from paper_2505_20968_gb300.binding import PRD
    P = PRD(_cfg(nnu, n_mu=2, n_chi=4, coherent=False), device=0)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 8, 0.1, 1.0)).to("cuda", torch.float32)
    for o in range(0, P.nO, 3):
        for s in range(4):
            y = torch.zeros_like(x)
            y[:, o, :, s] = x[:, o, :, s]
            ref = P.apply_sigma(y)
            for k in (-40, 30):
                d = P.apply_sigma(y * 2.0 ** k) * 2.0 ** -k - ref
                assert float(d.abs().max()) <= 1e-6 * float(ref.abs().max()), (o, s, k)
    P.device_status()
    P.close()
