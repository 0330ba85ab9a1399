"""The tensor-core contraction with its pipeline waits cut short at limits from one poll to many:
whichever wait gives up first, an apply either reports PRD_E_TIMEOUT or gives the emissivity of
an apply without a limit (5e-6 of each height's largest, the bound between the contraction's two
paths), and the context applies correctly afterwards.  One and two row blocks, packed tiles,
FP32 products and split-BF16 ones."""
import numpy as np
import pytest
import torch

from paper_2505_20968_gb300 import inputs

pytestmark = pytest.mark.gpu

E_TIMEOUT, OPT_WAIT_POLLS = -8, 3


def _worst(a, b):
    return max(np.max(np.abs(a[z] - b[z])) / np.max(np.abs(b[z, ..., 0])) for z in range(len(b)))


@pytest.mark.parametrize("nnu,contraction", [(27, "tf32x3"), (100, "tf32x3"), (150, "tf32x3"), (40, "bf16x3")])
def test_short_wait_limits_stop_cleanly(nnu, contraction):
    from paper_2505_20968_gb300.binding import PRD, lib
    P = PRD(inputs.hi_lya(n_z=4, n_core=nnu - 6, n_wing=6, n_mu_half=2, n_chi=4, seed=29), device=0)
    P.set_contraction(contraction)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 5, 0.1, 1.0)).to(P.device, P.dtype)
    ref = P.apply_sigma(x).cpu().numpy().astype(np.float64)
    P.device_status()
    for polls in (1, 2, 3, 8, 30, 100, 300, 1000, 3000, 10000):
        assert lib().prd_set_option(P.h, OPT_WAIT_POLLS, polls) == 0
        out = P.apply_sigma(x).cpu().numpy().astype(np.float64)
        rc = lib().prd_device_status(P.h)
        assert rc in (0, E_TIMEOUT)
        assert rc or _worst(out, ref) < 5e-6
        assert lib().prd_set_option(P.h, OPT_WAIT_POLLS, 0) == 0
        out = P.apply_sigma(x).cpu().numpy().astype(np.float64)
        P.device_status()
        assert _worst(out, ref) < 5e-6
    P.close()
