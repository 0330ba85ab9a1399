"""The tensor-core R_II contraction at the edges of its tiles: row counts either side of 32, 64
and 128 rows (tiles per pass, row blocks), of a 16-column K step, odd and even K-step counts
per half, and the largest count; direction counts from a handful to more than one record
of 32 entries; angle-averaged problems, whose outputs have all directions as partners; few work
items (their tiles split between CTAs, with incomplete last passes) and many.  Reference: the
CUDA-core contraction of the same context (the bound between the two paths in the parity
tests, 5e-6 of each height's largest emissivity; bf16 planes 1e-4, as there)."""
import numpy as np
import pytest
import torch

from paper_2505_20968_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cfg(nnu, n_z, n_mu, n_chi, mode):
    cfg = inputs.hi_lya(n_z=n_z, n_core=nnu - 6, n_wing=6, n_mu_half=n_mu, n_chi=n_chi, seed=41, mode=mode)
    return cfg


def _worst(a, b):
    return max(np.max(np.abs(a[z] - b[z])) / np.max(np.abs(b[z, ..., 0])) for z in range(len(b)))


@pytest.mark.parametrize("nnu,n_z,n_mu,n_chi,mode", [
    (9, 2, 1, 3, inputs.MODE_AD), (16, 2, 1, 4, inputs.MODE_AD), (17, 3, 2, 4, inputs.MODE_AD),
    (32, 4, 2, 5, inputs.MODE_AD), (33, 2, 2, 4, inputs.MODE_AD), (64, 2, 1, 3, inputs.MODE_AD),
    (65, 2, 2, 3, inputs.MODE_AD), (128, 2, 1, 4, inputs.MODE_AD), (129, 2, 2, 4, inputs.MODE_AD),
    (224, 2, 1, 3, inputs.MODE_AD), (40, 2, 4, 8, inputs.MODE_AD), (21, 2, 4, 8, inputs.MODE_AA),
    (70, 2, 3, 5, inputs.MODE_AA)])
def test_contraction_matches_the_cuda_core_path(nnu, n_z, n_mu, n_chi, mode):
    from paper_2505_20968_gb300.binding import PRD
    cfg = _cfg(nnu, n_z, n_mu, n_chi, mode)
    P = PRD(cfg, device=0)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 6, 0.1, 1.0)).to("cuda", torch.float32)
    P.set_tensor_cores(False)
    ref = P.apply_sigma(x).cpu().numpy().astype(np.float64)
    P.set_tensor_cores(True)
    out = P.apply_sigma(x).cpu().numpy().astype(np.float64)
    P.device_status()
    assert _worst(out, ref) < 5e-6
    # rows of very different size, and a zero one: the operand's scales are per direction and Stokes parameter
    x2 = x * torch.logspace(-30, 6, P.nO, device="cuda")[None, :, None, None]
    x2[:, 0, :, 1] = 0.0
    P.set_tensor_cores(False)
    ref = P.apply_sigma(x2).cpu().numpy().astype(np.float64)
    P.set_tensor_cores(True)
    assert _worst(P.apply_sigma(x2).cpu().numpy().astype(np.float64), ref) < 5e-6
    P.close()


@pytest.mark.parametrize("nnu,n_mu,n_chi", [(31, 2, 4), (64, 2, 4), (100, 1, 4), (150, 1, 4)])
def test_bf16_planes_match_fp32(nnu, n_mu, n_chi):
    from paper_2505_20968_gb300.binding import PRD
    cfg = _cfg(nnu, 2, n_mu, n_chi, inputs.MODE_AD)
    P, B = PRD(cfg, device=0), PRD(cfg, precision="fp32_bf16x3", device=0)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 6, 0.1, 1.0)).to("cuda", torch.float32)
    ref = P.apply_sigma(x).cpu().numpy().astype(np.float64)
    assert _worst(B.apply_sigma(x).cpu().numpy().astype(np.float64), ref) < 1e-4
    P.set_contraction("bf16x3")                    # FP32 tiles, re-split on the fly
    assert _worst(P.apply_sigma(x).cpu().numpy().astype(np.float64), ref) < 1e-4
    P.device_status()
    B.device_status()
    P.close()
    B.close()


def test_nan_and_infinite_inputs_stay_visible():
    from paper_2505_20968_gb300.binding import PRD
    P = PRD(_cfg(20, 2, 1, 3, inputs.MODE_AD), device=0)
    x = torch.ones(P.shape, device="cuda")
    for bad in (float("nan"), float("inf")):
        y = x.clone()
        y[1, 2, 7, 0] = bad
        e = P.apply_sigma(y)
        assert bool(torch.isfinite(e[0]).all()) and not bool(torch.isfinite(e[1]).all())
    P.close()
