"""The workspace of the tensor-core contraction: a small part of a context whatever the number of
directions and heights (at most 1 GiB, or one height), there before the FP64 copy of the tiles
is weighed against free memory; problems of more heights than it holds take several launches,
which agree with the CUDA-core contraction as one launch does (5e-6 of each height's largest
emissivity, the bound between the two paths)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2505_20968_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sizes_of_setup(cfg):
    """Sizes a context asks its allocator for, in order."""
    from paper_2505_20968_gb300 import binding as b
    sizes = []
    L = b.lib()

    def alloc(nbytes, user, stream):
        sizes.append(int(nbytes))
        return torch.cuda.caching_allocator_alloc(int(nbytes), device=0, stream=int(stream or 0))

    def free(ptr, user):
        torch.cuda.caching_allocator_delete(int(ptr))

    fa, ff = b._ALLOC_FN(alloc), b._FREE_FN(free)
    P = b.PRD(cfg, precision="fp32", device=0, setup=False)
    assert L.prd_set_allocator(P.h, fa, ff, None) == 0
    P.setup()
    P.close()
    return sizes


def test_workspace_comes_before_the_fp64_tiles():
    nz, nnu = 3, 100
    cfg = inputs.hi_lya(n_z=nz, n_core=nnu - 6, n_wing=6, n_mu_half=2, n_chi=4, seed=5, mode=inputs.MODE_AA)
    sizes = _sizes_of_setup(cfg)
    nO = 16
    entries = nz * nO * (nO // 2) * nnu * 16      # all directions as partners, two an entry, 16 bytes a row
    assert entries in sizes
    assert sizes.index(entries) < sizes.index(max(sizes))      # the FP64 tiles are the largest buffer


def test_heights_in_several_launches():
    from paper_2505_20968_gb300.binding import PRD
    nz, nnu, nO = 38, 224, 128
    per = nO * (nO // 2) * nnu * 16
    assert 1 < (1 << 30) // per < nz
    cfg = inputs.hi_lya(n_z=nz, n_core=nnu - 6, n_wing=6, n_mu_half=8, n_chi=8, seed=6, mode=inputs.MODE_AA)
    P = PRD(cfg, device=0)
    x = torch.from_numpy(inputs.seeded_vector(P.shape, 6, 0.1, 1.0)).to("cuda", torch.float32)
    out = P.apply_sigma(x)
    P.device_status()
    P.set_profiling(True)
    P.apply_sigma(x)
    assert P.stage_times()["S3_R2_contraction"][1] == 1          # one run of the stage, however many launches
    P.set_profiling(False)
    P.set_tensor_cores(False)
    ref = P.apply_sigma(x)
    for z in range(nz):
        assert float((out[z] - ref[z]).abs().max() / ref[z, ..., 0].abs().max()) < 5e-6, z
    P.close()
