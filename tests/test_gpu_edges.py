"""Frame changes, quadrature rows and line-of-sight contraction at the sizes where their
kernels can go wrong: the smallest frequency count, counts beside the 8-step
blocks of the spline recurrence and the 16-column tiles, direction counts that are no
multiple of the rows a CTA takes, and few or many rows (either side of the one-row rule).
FP64 mode against the oracle: the two sides' quadratures each agree with the exact integral
to ~1e-9 (the bound of the parity tests)."""
import numpy as np
import pytest
import torch

from paper_2505_20968_gb300 import inputs

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("n_z,n_x,n_mu,n_chi,mode", [
    (2, 4, 1, 3, inputs.MODE_AD), (3, 5, 2, 3, inputs.MODE_AD), (2, 10, 1, 4, inputs.MODE_AD),
    (2, 17, 1, 5, inputs.MODE_AD), (2, 11, 1, 3, inputs.MODE_AA), (102, 4, 1, 3, inputs.MODE_AD)])
def test_two_level_operator_at_the_edges(n_z, n_x, n_mu, n_chi, mode):
    from oracle.problem import Problem
    from paper_2505_20968_gb300.binding import PRD
    cfg = inputs.twolevel_slab(n_z=n_z, n_x=n_x, n_mu_half=n_mu, n_chi=n_chi, eps=1e-2)
    cfg["quad"]["mode"] = mode
    v = np.zeros((n_z, 3))
    v[:, 2] = np.linspace(-3.0, 4.0, n_z)          # moves the spline points off the nodes
    v[:, 0] = 1.0
    cfg = dict(cfg, atm=dict(cfg["atm"], v_kms=v))
    P = PRD(cfg, device=0)
    O = Problem(cfg)
    x = inputs.seeded_vector(P.shape, 3, 0.1, 1.0)
    assert _rel(P.apply_operator(torch.from_numpy(x).cuda()).cpu().numpy(), O.apply_A(x)) < 1e-8


@pytest.mark.parametrize("nnu,prec,mode", [(9, "fp64", inputs.MODE_AD), (16, "fp32", inputs.MODE_AD),
                                           (13, "fp32", inputs.MODE_AA)])
def test_emergent_profiles_of_a_two_term_atom(nnu, prec, mode):
    from oracle.problem import Problem
    from paper_2505_20968_gb300.binding import PRD
    cfg = inputs.hi_lya(n_z=3, n_core=nnu - 6, n_wing=6, n_mu_half=1, n_chi=4, seed=33, mode=mode)
    P = PRD(cfg, precision=prec, device=0)
    O = Problem(cfg)
    x = inputs.seeded_vector(P.shape, 4, 0.1, 1.0)
    mu, chi = [1.0, 0.35], [0.0, 0.9]
    e = P.emergent_stokes(torch.from_numpy(x).to("cuda", P.dtype), mu, chi).cpu().numpy()
    for i in range(2):
        # FP32: the emergent bound of the parity tests, 1e-5
        assert _rel(e[i], O.emergent(x, mu[i], chi[i])) < (1e-8 if prec == "fp64" else 1e-5)
